"""GPU parity of the double-float inter-body sum with tensor-core sums (Sec. 3.3): right-hand-side
counts around its chunks of 8, 16 and 32, bodies whose nodes leave ragged target and source tiles,
a sum long enough for several chunks of sources, and nearly touching bodies, which keep the
one-directional kernel; against the oracle and against the one-directional kernel."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ragged():
    require_gpu()
    from oracle import Problem
    wl = W.two_spheres(n_panels=7, gl_order=9, n_modes=33, k=3.0, eta=1.0)       # 2 x 2,079 nodes
    return gpu_solver(wl), Problem(wl)


@pytest.mark.parametrize("R", [3, 7, 8, 9, 16, 17, 32, 33, 65])
def test_dfx_sum(ragged, R):
    s, P = ragged
    sig = rand_c((P.N, R), 800 + R)
    ref = P.interbody(sig)
    top = np.abs(ref).max()
    got = s.interbody(sig, precision=2)
    assert np.abs(got - ref).max() < 1e-12 * top
    assert np.array_equal(got, s.interbody(sig, precision=2))        # whole-number sums: any order
    s.set_fp64_interbody_engine(0)
    one = s.interbody(sig, precision=2)
    s.set_fp64_interbody_engine(-1)
    assert np.abs(got - one).max() < 1e-12 * top


def test_dfx_constant_density(ragged):
    """Equal densities: every digit product of a column has one sign."""
    s, P = ragged
    sig = np.ones((P.N, 8)) * np.array([1.0, -1.0, 1j, 1 + 1j, 1 / 3, 0.999999, 2.0 ** -30, 7.7e-3])[None, :]
    ref = P.interbody(sig.astype(complex))
    got = s.interbody(sig.astype(complex), precision=2)
    assert (np.abs(got - ref).max(axis=0) < 1e-12 * np.abs(ref).max(axis=0)).all()


@pytest.mark.parametrize("gap", [0.3, 0.03])
def test_dfx_close_bodies(gap):
    """On both sides of the rule on the kernel's range (k = 2: ratios of about 27 and 1,200)."""
    require_gpu()
    from oracle import Problem
    wl = W.two_spheres(n_panels=7, gl_order=9, n_modes=33, sep=1.0 + gap / 2)
    s, P = gpu_solver(wl), Problem(wl)
    sig = rand_c((P.N, 8), 900)
    ref = P.interbody(sig)
    got = s.interbody(sig, precision=2)
    assert np.abs(got - ref).max() < 1e-12 * np.abs(ref).max()
    s.set_fp64_interbody_engine(0)
    assert np.array_equal(got, s.interbody(sig, precision=2)) == (gap < 0.1)
