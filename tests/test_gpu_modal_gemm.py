"""GPU parity of the CUDA-core mode GEMM inside D^{-1} (step (2) of the Remark after
Eq. (precond)) over its column widths (2, 4, 8, 16 and wider, with ragged last columns), rows
that do not fill the last block, and k sums in one tile and in several, in each precision,
against the oracle."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("panels,gl", [(3, 5), (4, 11), (9, 15), (13, 20)])
def test_local_inverse_columns(panels, gl):
    require_gpu()
    from oracle import Problem
    wl = W.two_spheres(n_panels=panels, gl_order=gl, n_modes=5)
    s, P = gpu_solver(wl), Problem(wl)
    s.set_modal_engine(0)
    y = rand_c((P.N, 19), 77)
    ref = P.local_inverse(y)
    top = np.abs(ref).max()
    for R in (1, 2, 3, 4, 8, 9, 19):
        for precision, tol in ((0, 1e-11), (2, 1e-11), (1, 1e-5)):
            got = s.local_inverse(np.ascontiguousarray(y[:, :R]), precision=precision)
            assert np.abs(got - ref[:, :R]).max() < tol * top, (R, precision)
