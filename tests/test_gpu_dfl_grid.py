"""The double-float sum on grids (one-directional, many sources and right-hand sides), which nearly
touching bodies and k = 0 still take and the explicit engine 0 selects: columns of very different sizes,
a zero column, nodes over eight decades, NaN and infinity, ragged chunks of right-hand sides and long
sums, against the oracle."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def spheres():
    require_gpu()
    from oracle import Problem
    wl = W.two_spheres()                             # 4,100 sources of every target
    s = gpu_solver(wl)
    s.set_fp64_interbody_engine(0)
    return s, Problem(wl)


@pytest.mark.parametrize("R", [5, 8, 9, 17, 33])
def test_many_sources(spheres, R):
    s, P = spheres
    sig = rand_c((P.N, R), 300 + R)
    ref = P.interbody(sig)
    assert np.abs(s.interbody(sig, precision=2) - ref).max() < 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("R", [8, 16, 20])
def test_scales(spheres, R):
    s, P = spheres
    sig = rand_c((P.N, R), 500 + R) * 10.0 ** np.linspace(-8, 0, P.N)[:, None]
    sig *= 10.0 ** np.linspace(-150, 150, R)[None, :]
    sig[:, 1] = 0.0
    got, ref = s.interbody(sig, precision=2), P.interbody(sig)
    assert (np.abs(got - ref).max(axis=0) <= 1e-12 * np.abs(ref).max(axis=0)).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite(spheres, bad):
    s, P = spheres
    sig = rand_c((P.N, 8), 708)
    sig[17, 0] = bad
    got, n = s.interbody(sig, precision=2), P.N // 2
    assert not np.isfinite(got[n:, 0]).any() and np.isfinite(got[:n]).all()
    ref = P.interbody(sig[:, 1:])
    assert np.abs(got[:, 1:] - ref).max() < 1e-12 * np.abs(ref).max()


def test_equal_densities(spheres):
    """Every term of a tile at its grid's limit with one sign."""
    s, P = spheres
    sig = np.ones((P.N, 8), complex) * np.array([1, -1, 1j, 1 + 1j, 1 / 3, 0.999999, 2.0 ** -30, 7.7e-3])[None, :]
    ref = P.interbody(sig)
    got = s.interbody(sig, precision=2)
    assert (np.abs(got - ref).max(axis=0) < 1e-12 * np.abs(ref).max(axis=0)).all()


def test_default_route_of_close_bodies():
    """Nearly touching bodies with many sources: automatic and engine 0 are one kernel."""
    require_gpu()
    from oracle import Problem
    wl = W.two_spheres(sep=1.01)
    s, P = gpu_solver(wl), Problem(wl)
    sig = rand_c((P.N, 8), 710)
    got, ref = s.interbody(sig, precision=2), P.interbody(sig)
    assert np.abs(got - ref).max() < 1e-12 * np.abs(ref).max()
    s.set_fp64_interbody_engine(0)
    assert np.array_equal(got, s.interbody(sig, precision=2))
