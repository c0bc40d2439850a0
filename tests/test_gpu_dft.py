"""GPU parity of the folded azimuthal DFTs inside D^{-1} (steps (1) and (3) of the Remark after
Eq. (precond)) at the smallest mode counts, odd and prime ones, and every blocking of the
right-hand sides (1, 2 and 3, 4 and more with a ragged last block), in each precision,
against the oracle."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("modes", [3, 5, 9, 37])
@pytest.mark.parametrize("R", [1, 2, 3, 4, 7, 17])
def test_local_inverse_folded(modes, R):
    require_gpu()
    from oracle import Problem
    wl = W.two_spheres(n_panels=3, gl_order=5, n_modes=modes)
    s, P = gpu_solver(wl), Problem(wl)
    y, sig = rand_c((P.N, R), 900 + R), rand_c((P.N, R), 950 + R)
    ref = P.local_inverse(y)
    top = np.abs(ref).max()
    for precision, tol in ((0, 1e-11), (2, 1e-11), (1, 1e-5)):
        assert np.abs(s.local_inverse(y, precision=precision) - ref).max() < tol * top, precision
        got = s.local_inverse(y, sigma=sig, alpha=0.5, beta=-2.0, precision=precision)
        assert np.abs(got - (0.5 * sig - 2.0 * ref)).max() < 2 * tol * top + 1e-15, precision
