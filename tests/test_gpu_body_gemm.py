"""GPU parity of the product with one matrix per body shape that the accelerated scheme's local
operator, restriction and extension share (Sec. 5), at column counts (bodies x right-hand sides)
that fill one to four lane groups and leave ragged ones, and at row counts around the blocks'
rows and the staged terms, in each precision, against the oracle."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, rel_l2, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,R", [(1, 1), (63, 1), (65, 2), (128, 4), (130, 5), (257, 6), (33, 17)])
def test_reduced_operator_columns(k, R):
    require_gpu()
    from oracle import Problem
    from oracle.compress import Compressed
    wl = W.separated_spheroids(spacing=4.0, n_panels=6, gl_order=8, n_modes=9)
    P = Problem(wl)
    shp = wl.bodies[0].shape
    g = np.random.default_rng(1000 + k)
    J = np.sort(g.choice(shp.n_nodes, k, replace=False))
    T = (g.standard_normal((k, shp.n_nodes)) + 1j * g.standard_normal((k, shp.n_nodes))) / np.sqrt(shp.n_nodes)
    T[:, J] = np.eye(k)
    C = Compressed(P, 0.0, skeletons={shp: (J, T)})
    s = gpu_solver(wl)
    s.set_skeleton(0, J, T)
    sig = rand_c((C.Nk, R), 40 + R)
    ref = C.apply(sig)
    top = np.abs(ref).max()
    assert np.abs(s.apply_reduced(sig, precision=0) - ref).max() < 1e-12 * top
    assert np.abs(s.apply_reduced(sig, precision=2) - ref).max() < 1e-11 * top
    assert rel_l2(s.apply_reduced(sig, precision=1), ref) < 5e-6
