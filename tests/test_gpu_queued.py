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


def test_timeout_in_the_reduced_system(monkeypatch):
    """The accelerated scheme's operator (host data) reports a wait that ran out in its own sums."""
    require_gpu()
    from paper_1406_0236_gb300 import HzbError
    from tests._common import gpu_solver
    monkeypatch.setenv("HZB_FAULT", "timeout")
    wl = W.separated_spheroids(spacing=4.0, n_panels=6, gl_order=8, n_modes=9)
    n, k = wl.bodies[0].shape.n_nodes, 257
    g = np.random.default_rng(3)
    J = np.sort(g.choice(n, k, replace=False))
    T = (g.standard_normal((k, n)) + 1j * g.standard_normal((k, n))) / np.sqrt(n)
    T[:, J] = np.eye(k)
    s = gpu_solver(wl)
    s.set_skeleton(0, J, T)
    x = rand_c((3 * k, 48), 6)                       # 2.9e7 pairs times right-hand sides
    with pytest.raises(HzbError) as e:
        s.apply_reduced(x, precision=2)
    assert e.value.status == -6
    ref = s.apply_reduced(x, precision=0)
    assert np.abs(s.apply_reduced(x, precision=2) - ref).max() < 1e-11 * np.abs(ref).max()
