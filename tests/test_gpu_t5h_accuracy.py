"""Where the automatic FP32 sum takes the tensor cores, its error against FP64 is no larger than that of
the packed FP32 kernel, which it replaced there (Sec. 3.3)."""
import numpy as np
import pytest

import workloads as W
from tests._common import rand_c, rel_l2, require_gpu

pytestmark = pytest.mark.gpu


# small k, where the phase error does not hide the sums'
@pytest.mark.parametrize("k,R", [(1.0, 12), (2.0, 9), (2.0, 12), (2.0, 15), (2.0, 24)])
def test_error_against_packed_kernel(k, R):
    require_gpu()
    from paper_1406_0236_gb300 import Options, Solver
    s = Solver.from_workload(W.two_spheres(k=k), Options())
    sig = rand_c((s.N, R), 60 + R)
    ref = s.interbody(sig)
    err = {}
    for engine in (-1, 3):
        s.set_interbody_engine(engine)
        err[engine] = rel_l2(s.interbody(sig, precision=1), ref)
    assert err[-1] <= err[3]
