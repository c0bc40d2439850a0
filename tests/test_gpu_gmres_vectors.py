"""GPU solves through the GMRES vector kernels (dot products, updates, rotations, back
substitution) at right-hand-side counts around their blocks (1, 3, 31, 32, 33, 65), with and
without restarts, and with more than 32 basis vectors, against the oracle's dense solve."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, rel_l2, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def small():
    require_gpu()
    from oracle import Problem
    wl = W.two_spheres(n_panels=3, gl_order=6, n_modes=7)
    P = Problem(wl)
    return wl, P.N, P.dense_matrix()


@pytest.mark.parametrize("R,restart", [(1, 0), (3, 8), (31, 0), (32, 9), (33, 0), (65, 0)])
def test_solve_against_dense(small, R, restart):
    wl, N, D = small
    v = rand_c((N, R), 60 + R)
    s = gpu_solver(wl, tol=1e-12, restart=restart, maxit=400)
    assert s.solve_data(v).converged
    ref = np.linalg.solve(D, -v)
    got = s.get_density()
    for r in range(R):
        assert rel_l2(got[:, r], ref[:, r]) < 1e-9


def test_more_than_32_basis_vectors(small):
    """Random data on a small system takes more than a warp of basis vectors in one cycle."""
    wl, N, D = small
    v = rand_c((N, 2), 99)
    s = gpu_solver(wl, tol=1e-15, maxit=48)
    try:
        s.solve_data(v, allow_noconv=True)
    except Exception:
        pass
    ref = np.linalg.solve(D, -v)
    got = s.get_density()
    assert rel_l2(got, ref) < 1e-9
