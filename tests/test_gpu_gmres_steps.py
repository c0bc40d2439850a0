"""GMRES over more basis vectors than a warp has lanes, with the number of steps checked, and at sizes
where the update of a step takes more than one block per SM."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, rel_l2, require_gpu

pytestmark = pytest.mark.gpu


def test_more_than_32_steps():
    """Six nearly touching spheres take 53 steps to 1e-14 in one cycle."""
    require_gpu()
    from oracle import Problem
    shape = W.ShapeSpec(W.SPHERE, (1.0,), 3, 5, 11)
    bodies = [W.Body(shape, 2.1 * np.array([q % 2, q // 2 % 2, q // 4], float), np.eye(3)) for q in range(6)]
    wl = W.Workload("six", bodies, 4.0, 4.0, np.array([[0, 0, 1.0]]))
    P = Problem(wl)
    v = rand_c((P.N, 2), 98)
    s = gpu_solver(wl, tol=1e-13, maxit=100)
    st = s.solve_data(v)
    assert st.converged and st.iterations > 32
    assert rel_l2(s.get_density(), np.linalg.solve(P.dense_matrix(), -v)) < 1e-9


@pytest.mark.parametrize("R", [16, 33])
def test_many_blocks(R):
    """40,400 unknowns: the residual of every right-hand side by the FP64 operator."""
    require_gpu()
    s = gpu_solver(W.two_spheres(n_panels=20, gl_order=10, n_modes=101), precision=1, tol=1e-9, residual=2)
    v = rand_c((s.N, R), 97)
    assert s.solve_data(v).converged
    sig = s.get_density()
    cols = [0, R // 2, R - 1]
    b = -s.local_inverse(np.ascontiguousarray(v[:, cols]))
    res = b - s.apply(np.ascontiguousarray(sig[:, cols]))
    assert (np.linalg.norm(res, axis=0) < 2e-9 * np.linalg.norm(b, axis=0)).all()
