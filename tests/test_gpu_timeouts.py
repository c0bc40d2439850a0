"""The bounded-wait exits of the tensor-core kernels that every default call uses, entered through a
flag the host sets before the launch: the mode GEMM of D^{-1} gives up with copies and MMAs in
flight, the double-float sum (alone and as pairs of CTAs) before it issues any.  Each reports
HZB_ETIMEOUT, and the same context then gives the right result."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, rel_l2, require_gpu

pytestmark = pytest.mark.gpu

ETIMEOUT = -6


def _times_out(call):
    from paper_1406_0236_gb300 import HzbError
    with pytest.raises(HzbError) as e:
        call()
    assert e.value.status == ETIMEOUT


@pytest.mark.parametrize("panels,gl,modes,R", [(3, 5, 9, 3), (10, 10, 41, 16)])
def test_modal_gemm_timeout(monkeypatch, panels, gl, modes, R):
    """One chunk of the k sum in flight, and several with both stages and accumulators taken."""
    require_gpu()
    monkeypatch.setenv("HZB_FAULT", "timeout_modal")
    wl = W.two_spheres(n_panels=panels, gl_order=gl, n_modes=modes)
    s = gpu_solver(wl)
    s.set_modal_engine(2)
    y = rand_c((s.N, R), 21)
    ref = s.local_inverse(y)
    _times_out(lambda: s.local_inverse(y, precision=1))
    assert rel_l2(s.local_inverse(y, precision=1), ref) < 1e-5


@pytest.mark.parametrize("R", [8, 16, 32, 33])
def test_double_float_sum_timeout(monkeypatch, R):
    require_gpu()
    monkeypatch.setenv("HZB_FAULT", "timeout")
    wl = W.two_spheres(n_panels=7, gl_order=9, n_modes=33)
    s = gpu_solver(wl)
    sig = rand_c((s.N, R), 22)
    ref = s.interbody(sig)
    _times_out(lambda: s.interbody(sig, precision=2))
    assert np.abs(s.interbody(sig, precision=2) - ref).max() < 1e-12 * np.abs(ref).max()
