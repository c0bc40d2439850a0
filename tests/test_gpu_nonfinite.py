"""A NaN or an infinity in one node of one right-hand side reaches everything that depends on it, in
its own column alone, through every engine of the FP32 mode GEMM and of the FP32 inter-body sum
(the TF32 engines round on the bit pattern, where a NaN is easily lost)."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, rel_l2, require_gpu

pytestmark = pytest.mark.gpu

BAD = [np.nan, np.inf, complex(0.0, np.nan), complex(1.0, -np.inf)]


@pytest.mark.parametrize("engine", [0, 1, 2])
@pytest.mark.parametrize("bad", BAD)
def test_local_inverse_not_finite(engine, bad):
    require_gpu()
    wl = W.two_spheres(n_panels=4, gl_order=8, n_modes=9)
    s = gpu_solver(wl)
    y = rand_c((s.N, 9), 31)
    ref = s.local_inverse(y)
    y[17, 2] = bad
    s.set_modal_engine(engine)
    got = s.local_inverse(y, precision=1)
    n = s.N // 2
    assert not np.isfinite(got[:n, 2]).any() and np.isfinite(got[n:, 2]).all()
    rest = [c for c in range(9) if c != 2]
    assert rel_l2(got[:, rest], ref[:, rest]) < 1e-5


@pytest.mark.parametrize("engine,k", [(1, 2.0), (2, 2.0), (3, 2.0), (4, 2.0), (5, 2.0), (5, 0.0), (6, 2.0), (7, 2.0)])
@pytest.mark.parametrize("bad", BAD)
def test_sum_not_finite(engine, k, bad):
    require_gpu()
    from paper_1406_0236_gb300 import Options, Solver
    s = Solver.from_workload(W.two_spheres(n_panels=4, gl_order=8, n_modes=9, k=k, eta=1.5), Options())
    sig = rand_c((s.N, 16), 32)
    ref = s.interbody(sig)
    sig[17, 2] = bad
    s.set_interbody_engine(engine)
    got = s.interbody(sig, precision=1)
    n = s.N // 2
    assert not np.isfinite(got[n:, 2]).any() and np.isfinite(got[:n, 2]).all()
    rest = [c for c in range(16) if c != 2]
    assert rel_l2(got[:, rest], ref[:, rest]) < (2e-3 if engine == 7 else 5e-6)
