"""GPU parity of the FP16 three-term tensor-core form of the FP32 inter-body sum (Sec. 3.3):
ragged tiles, bodies and right-hand-side chunks, source chunks, columns of very different
sizes, a NaN, and geometries outside its range (which take the TF32 form), against the oracle."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, rel_l2, require_gpu

pytestmark = pytest.mark.gpu


def _pair(n_panels, gl, modes, n_bodies=2, sep=3.0, k=2.5, eta=2.5):
    shape = W.ShapeSpec(W.SPHERE, (1.0,), n_panels, gl, modes)
    bodies = [W.Body(shape, np.array([sep * q, 0.0, 0.0]), np.eye(3)) for q in range(n_bodies)]
    return W.Workload("pair", bodies, k, eta, np.array([[0, 0, 1.0]]))


def _solver(wl):
    from oracle import Problem
    from paper_1406_0236_gb300 import Options, Solver
    s = Solver.from_workload(wl, Options())
    s.set_interbody_engine(5)
    return s, Problem(wl)


# nodes per body: 45 (two tiles, one ragged), 231, 513 (a block of one target), 1,300 x 4
@pytest.mark.parametrize("size", [(3, 5, 3, 2), (3, 7, 11, 2), (3, 9, 19, 2), (10, 10, 13, 4)])
@pytest.mark.parametrize("R", [1, 5, 16, 17, 33])
def test_t5h_sizes(size, R):
    require_gpu()
    s, P = _solver(_pair(*size))
    sig = rand_c((P.N, R), 800 + R)
    assert rel_l2(s.interbody(sig, precision=1), P.interbody(sig)) < 2e-6


# k r up to 50: the phase alone, k r times the rounding of r, is 2.0e-6 in the TF32 kernels
FAR = 3e-6


def test_t5h_uneven_bodies():
    require_gpu()
    s, P = _solver(W.uneven3())
    sig = rand_c((P.N, 20), 820)
    assert rel_l2(s.interbody(sig, precision=1), P.interbody(sig)) < FAR


def test_t5h_column_sizes_and_nan():
    require_gpu()
    s, P = _solver(W.uneven3())
    sig = rand_c((P.N, 18), 830) * 10.0 ** np.linspace(-30, 30, 18)[None, :]
    sig[:, 3] = 0.0
    ref, got = P.interbody(sig), s.interbody(sig, precision=1)
    for r in range(18):
        assert np.linalg.norm(got[:, r] - ref[:, r]) <= FAR * np.linalg.norm(ref[:, r])
    sig[5, 2] = np.nan
    got = s.interbody(sig, precision=1)
    n0 = P.N - np.count_nonzero(np.isnan(got[:, 2]))       # rows of the NaN's own body
    assert 0 < n0 < P.N and np.isfinite(np.delete(got, 2, axis=1)).all()


@pytest.mark.parametrize("wl", [dict(k=0.0, eta=1.5), dict(eta=0.0), dict(eta=-2.5), dict(sep=2.0004),
                                dict(n_bodies=3, sep=2.02)])
def test_t5h_range(wl):
    """k = 0, eta = 0 and bodies that nearly touch are outside FP16's range."""
    require_gpu()
    s, P = _solver(_pair(4, 6, 9, **wl))
    sig = rand_c((P.N, 16), 840)
    ref = P.interbody(sig)
    assert np.abs(s.interbody(sig, precision=1) - ref).max() < 3e-6 * np.abs(ref).max()
