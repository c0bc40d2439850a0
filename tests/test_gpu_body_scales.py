"""Inter-body sums of densities that differ by orders of magnitude from body to body (Sec. 3.3).  The
rows of a body sum the other bodies' densities only: those scaled by a power of two, the body's rows
scale with them bit for bit, however large its own densities are."""
import numpy as np
import pytest

import workloads as W
from tests._common import gpu_solver, rand_c, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def three():
    require_gpu()
    wl = W.uneven3()
    return gpu_solver(wl), np.cumsum([0] + [b.shape.n_nodes for b in wl.bodies])


def _rows_scale(three, R, exponent, call):
    s, off = three
    sig = rand_c((s.N, R), 70 + R)
    ref = call(sig)
    for a, b in zip(off[:-1], off[1:]):
        x = sig * 2.0 ** exponent
        x[a:b] = sig[a:b]
        x[:, 1] = sig[:, 1]                          # one column as it was
        got = call(x)
        want = ref[a:b] * 2.0 ** exponent
        want[:, 1] = ref[a:b, 1]
        assert np.array_equal(got[a:b], want), (a, np.abs(got[a:b] - want).max() / np.abs(want).max())


@pytest.mark.parametrize("exponent", [-20, -40, -80, 30])
@pytest.mark.parametrize("R", [5, 16, 20])
@pytest.mark.parametrize("engine", [5, 3])
def test_fp32_sum(three, engine, R, exponent):
    s = three[0]
    s.set_interbody_engine(engine)
    try:
        _rows_scale(three, R, exponent, lambda x: s.interbody(x, precision=1))
    finally:
        s.set_interbody_engine(-1)
