"""GPU parity of the far field and the exterior field for every width of the point kernels
(one block per point up to four right-hand sides, tiles of 8, 16, 32 and 64 columns above),
over ragged point and source tiles, against the oracle's sums of the same densities."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rel_l2, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,T", [(1, 1), (2, 5), (3, 17), (5, 33), (9, 16), (17, 2), (33, 15), (65, 31)])
def test_point_fields(R, T):
    require_gpu()
    from oracle import Problem, fields
    wl = W.tiny_two_spheres()
    s, P = gpu_solver(wl), Problem(wl)
    s.solve_plane_waves(W.uniform_directions(R, 3))
    sig = s.get_density()
    xh, pts = W.uniform_directions(T, 4), W.exterior_targets(wl, T, 5)
    far = np.stack([fields.far_field(P.nodes, sig[:, r], P.k, P.eta, xh) for r in range(R)], axis=1)
    near = np.stack([fields.field(P.nodes, sig[:, r], P.k, P.eta, pts) for r in range(R)], axis=1)
    assert rel_l2(s.far_field(xh), far) <= 1e-13
    assert rel_l2(s.eval_field(pts), near) <= 1e-13
