"""GPU parity of the pair-symmetric inter-body sums (Sec. 3.3) where several CTAs share a
block pair: the source side of a pair cut into runs of tiles, down to one tile, and the
rotation steps of a tile shared out, over ragged blocks and tiles, against the oracle."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, rel_l2, require_gpu

pytestmark = pytest.mark.gpu


def _pair(n_panels, gl, modes, n_bodies=2):
    shape = W.ShapeSpec(W.SPHERE, (1.0,), n_panels, gl, modes)
    bodies = [W.Body(shape, np.array([3.0 * q, 0.2 * q, -0.1 * q]), np.eye(3)) for q in range(n_bodies)]
    return W.Workload("pair", bodies, 2.5, 2.5, np.array([[0, 0, 1.0]]))


# nodes per body: 45 (a ragged second tile), 231, 513 (a last block of one node), 1,300 x 4
SIZES = [(3, 5, 3, 2), (3, 7, 11, 2), (3, 9, 19, 2), (10, 10, 13, 4)]


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("R", [1, 2, 3])
def test_shared_block_pairs(size, R):
    require_gpu()
    from oracle import Problem
    wl = _pair(*size)
    s, P = gpu_solver(wl), Problem(wl)
    sig = rand_c((P.N, R), 71 + R)
    ref = P.interbody(sig)
    s.set_interbody_engine(4)                   # pair-symmetric also for R = 3
    try:
        for precision, tol in ((0, 1e-12), (2, 1e-12)):
            got = s.interbody(sig, precision=precision)
            assert np.abs(got - ref).max() < tol * np.abs(ref).max(), (size, R, precision)
        assert rel_l2(s.interbody(sig, precision=1), ref) < 2e-6
    finally:
        s.set_interbody_engine(-1)


@pytest.mark.parametrize("k,eta", [(0.0, 1.5), (2.5, 0.0), (1e-9, 1.0), (3.0, 1e-9), (2.5, -2.5)])
def test_every_wave_and_coupling(k, eta):
    """The kernels scale lengths and normals by k and k / eta where both are in range; the
    others, a static kernel and a pure double layer among them, take the unscaled form."""
    require_gpu()
    from oracle import Problem
    from paper_1406_0236_gb300 import Options, Solver
    wl = W.two_spheres(n_panels=4, gl_order=7, n_modes=13, k=k, eta=eta)
    s, P = Solver.from_workload(wl, Options()), Problem(wl)
    for R in (1, 2, 4):
        sig = rand_c((P.N, R), 91 + R)
        ref = P.interbody(sig)
        s.set_interbody_engine(4)
        assert np.abs(s.interbody(sig) - ref).max() < 1e-12 * np.abs(ref).max(), R
        assert rel_l2(s.interbody(sig, precision=1), ref) < 2e-6, R
