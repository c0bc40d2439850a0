"""The automatic engine of the FP32 inter-body sum depends on the geometry and the sizes alone, not on
what the context ran before: a double-float sum, which looks at the geometry, changes nothing."""
import numpy as np
import pytest

import workloads as W
from tests._common import rand_c, require_gpu

pytestmark = pytest.mark.gpu


# k = 0, nearly touching bodies (both outside FP16's range), an ordinary pair; below and above the
# pair work from which on the tensor cores take 16 right-hand sides
@pytest.mark.parametrize("case", [dict(k=0.0, eta=1.5), dict(sep=1.0002), dict()])
@pytest.mark.parametrize("modes,R", [(33, 16), (33, 8), (41, 16)])
def test_choice_does_not_depend_on_earlier_calls(case, modes, R):
    require_gpu()
    from paper_1406_0236_gb300 import Options, Solver
    s = Solver.from_workload(W.two_spheres(n_panels=7, gl_order=9, n_modes=modes, **case), Options())
    sig = rand_c((s.N, R), 50 + R)
    first = s.interbody(sig, precision=1)
    s.interbody(np.ascontiguousarray(sig[:, :8]), precision=2)
    assert np.array_equal(first, s.interbody(sig, precision=1))
