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


@pytest.mark.parametrize("exponent", [-20, -40, 30])
@pytest.mark.parametrize("R", [3, 8, 16, 33])
@pytest.mark.parametrize("engine", [-1, 0])
def test_double_float_sum(three, engine, R, exponent):
    s = three[0]
    s.set_fp64_interbody_engine(engine)
    try:
        _rows_scale(three, R, exponent, lambda x: s.interbody(x, precision=2))
    finally:
        s.set_fp64_interbody_engine(-1)


def test_double_float_chain():
    """Bodies at 1, 1e-9 and 1e-18 with an odd number of tiles each, so that pairs of tiles end with a
    body: the rows of every body against the FP64 sum, by their own largest value."""
    require_gpu()
    shape = W.ShapeSpec(W.SPHERE, (1.0,), 5, 11, 29)           # 1,595 nodes, 50 tiles, the last ragged
    other = W.ShapeSpec(W.SPHERE, (0.8,), 5, 10, 21)           # 1,050 nodes, 33 tiles
    bodies = [W.Body(sh, np.array([3.0 * q, 0.3 * q, 0.0]), np.eye(3)) for q, sh in enumerate((other, shape, other))]
    s = gpu_solver(W.Workload("chain", bodies, 2.0, 2.0, np.array([[0, 0, 1.0]])))
    off = np.cumsum([0] + [b.shape.n_nodes for b in bodies])
    for R in (8, 33):
        for order in ([0, 1, 2], [2, 1, 0], [1, 2, 0]):
            sig = rand_c((s.N, R), 90 + R)
            for q in range(3):
                sig[off[q]:off[q + 1]] *= 1e-9 ** order[q]
            ref, got = s.interbody(sig), s.interbody(sig, precision=2)
            for a, b in zip(off[:-1], off[1:]):
                assert (np.abs(got[a:b] - ref[a:b]).max(axis=0) < 1e-12 * np.abs(ref[a:b]).max(axis=0)).all(), (R, order, a)
