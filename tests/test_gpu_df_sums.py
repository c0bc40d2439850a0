"""GPU parity of the double-float inter-body sum (Sec. 3.3) over its routes: the
pair-symmetric kernel, the one-directional kernel with two-sums (few sources or few
right-hand sides) and with sums on a grid (many of both), ragged right-hand-side chunks,
densities of very different sizes, k = 0, and a NaN, against the oracle."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, require_gpu

pytestmark = pytest.mark.gpu


def _solver(wl):
    from oracle import Problem
    return gpu_solver(wl), Problem(wl)


@pytest.fixture(scope="module")
def spheres():
    require_gpu()
    return _solver(W.two_spheres())                  # 4,100 sources of every target


@pytest.mark.parametrize("R", [1, 2, 3, 5, 8, 9, 17, 33])
def test_df_sum_many_sources(spheres, R):
    s, P = spheres
    sig = rand_c((P.N, R), 300 + R)
    ref = P.interbody(sig)
    assert np.abs(s.interbody(sig, precision=2) - ref).max() < 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("R", [3, 4, 6, 16, 20])
def test_df_sum_few_sources(R):
    require_gpu()
    s, P = _solver(W.uneven3())
    sig = rand_c((P.N, R), 400 + R)
    ref = P.interbody(sig)
    for engine in (-1, 0, 1):
        s.set_fp64_interbody_engine(engine)
        assert np.abs(s.interbody(sig, precision=2) - ref).max() < 1e-12 * np.abs(ref).max(), engine


@pytest.mark.parametrize("R", [2, 8])
def test_df_sum_scales(spheres, R):
    """Columns from 1e-150 to 1e150, a zero column, and nodes over eight decades."""
    s, P = spheres
    sig = rand_c((P.N, R), 500 + R) * 10.0 ** np.linspace(-8, 0, P.N)[:, None]
    sig *= 10.0 ** np.linspace(-150, 150, R)[None, :]
    if R > 2:
        sig[:, 1] = 0.0
    got, ref = s.interbody(sig, precision=2), P.interbody(sig)
    top = np.abs(ref).max(axis=0)
    assert (np.abs(got - ref).max(axis=0) <= 1e-12 * top).all()


@pytest.mark.parametrize("R", [1, 4, 8])
def test_df_sum_k_zero(R):
    require_gpu()
    wl = W.two_spheres(n_panels=6, gl_order=8, n_modes=21, k=0.0, eta=1.5)
    from oracle import Problem
    from paper_1406_0236_gb300 import Options, Solver
    s, P = Solver.from_workload(wl, Options()), Problem(wl)
    sig = rand_c((P.N, R), 600 + R)
    ref = P.interbody(sig)
    assert np.abs(s.interbody(sig, precision=2) - ref).max() < 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("R", [1, 8])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_df_sum_not_finite(spheres, R, bad):
    """A NaN or an infinity reaches every target of the other body, in its own column alone."""
    s, P = spheres
    sig = rand_c((P.N, R), 700 + R)
    sig[17, 0] = bad
    got = s.interbody(sig, precision=2)
    n = P.N // 2
    assert not np.isfinite(got[n:, 0]).any() and np.isfinite(got[:n]).all()
    if R > 1:
        ref = P.interbody(sig[:, 1:])
        assert np.abs(got[:, 1:] - ref).max() < 1e-12 * np.abs(ref).max()
