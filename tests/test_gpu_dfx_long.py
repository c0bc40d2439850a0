"""Double-float inter-body sums whose chunks of sources are longer than the 256 tiles that the
64-bit sums hold (Sec. 3.3): right-hand sides of one CTA and of a pair of CTAs, with a ragged last
tile, against the FP64 sum; and the memory that a large sum takes."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, require_gpu

pytestmark = pytest.mark.gpu


def _spheroids(n_panels, gl, modes):
    from paper_1406_0236_gb300 import Options, Solver
    wl = W.spheroids8(n_panels=n_panels, gl_order=gl, n_modes=modes)
    return Solver.from_workload(wl, Options())


# 8 x 9,090 nodes: 1,995 source tiles of a target, in five chunks for R = 3
@pytest.mark.parametrize("R,cols", [(3, [0, 1, 2]), (33, [0, 17, 32])])
def test_long_chunks(R, cols):
    require_gpu()
    s = _spheroids(9, 10, 101)
    sig = rand_c((s.N, R), 950 + R)
    ref = s.interbody(np.ascontiguousarray(sig[:, cols]))
    got = s.interbody(sig, precision=2)
    assert np.abs(got[:, cols] - ref).max() < 1e-12 * np.abs(ref).max()
    assert np.array_equal(got, s.interbody(sig, precision=2))


def test_long_chunk_not_finite():
    require_gpu()
    s = _spheroids(9, 10, 101)
    sig = rand_c((s.N, 3), 960)
    sig[s.N - 5, 1] = np.nan
    got = s.interbody(sig, precision=2)
    n = s.N // 8 * 7
    assert np.isnan(got[:n, 1]).all() and np.isfinite(got[n:]).all()
    assert np.isfinite(got[:, [0, 2]]).all()


def test_large_sum_memory():
    """258,560 unknowns, 64 right-hand sides: the digit images are 0.8 GB."""
    require_gpu()
    import torch
    s = _spheroids(20, 16, 101)
    x = torch.zeros((s.N, 64), dtype=torch.complex128, device="cuda")
    x[::7] = 1.0
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    y = s.interbody(x, precision=2)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    assert bool(torch.isfinite(torch.view_as_real(y)).all())
    assert used < 2.5e9                              # (0.3 GB of it the result, and torch's own)
