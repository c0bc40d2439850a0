"""Sums on device data are queued on the context's stream: a caller's stream capture takes them, the
replays follow the input, and a bounded wait that ran out is reported by the next call that waits."""
import numpy as np
import pytest

import workloads as W
from tests._common import rand_c, require_gpu

pytestmark = pytest.mark.gpu


def _solver(stream):
    from paper_1406_0236_gb300 import Options, Solver
    return Solver.from_workload(W.two_spheres(), Options(), stream=stream.cuda_stream)


# precision 1: FP32 on the tensor cores (N^2 R >= 3e8); 2: double-float on the tensor cores
@pytest.mark.parametrize("precision,R", [(1, 9), (2, 3), (2, 16), (2, 33)])
def test_captured_sum(precision, R):
    require_gpu()
    import torch
    st = torch.cuda.Stream()
    s = _solver(st)
    a, b = (torch.tensor(rand_c((s.N, R), q), device="cuda") for q in (1, 2))
    x = a.clone()
    with torch.cuda.stream(st):
        want = s.interbody(b, precision=precision)
        s.interbody(x, precision=precision)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        y = s.interbody(x, precision=precision)
    x.copy_(b)
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(y), torch.view_as_real(want))


def test_timeout_of_a_queued_sum(monkeypatch):
    require_gpu()
    import torch
    from paper_1406_0236_gb300 import HzbError
    monkeypatch.setenv("HZB_FAULT", "timeout")
    st = torch.cuda.Stream()
    s = _solver(st)
    host = rand_c((s.N, 8), 5)
    with torch.cuda.stream(st):
        x = torch.tensor(host, device="cuda")
        y = s.interbody(x, precision=2)
    torch.cuda.synchronize()
    assert bool(torch.isnan(torch.view_as_real(y)).all())
    with pytest.raises(HzbError) as e:
        s.interbody(host, precision=2)               # host data: waits and reports
    assert e.value.status == -6
    ref = s.interbody(host, precision=0)
    assert np.abs(s.interbody(host, precision=2) - ref).max() < 1e-12 * np.abs(ref).max()
