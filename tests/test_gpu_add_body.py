"""A body added after a query or a sum has generated the nodes: the next calls see all bodies, in every
precision, as a context does that got them at once."""
import numpy as np
import pytest

import workloads as W
from tests._common import rand_c, require_gpu

pytestmark = pytest.mark.gpu


def _solver():
    from paper_1406_0236_gb300 import Options, Solver
    s = Solver(2.0, 2.0, Options())
    return s


def _add(s, q):
    s.add_body(W.SPHERE, (1.0,), 7, 9, 33, np.array([3.0 * q, 0.1 * q, 0.0]), np.eye(3))


def test_body_added_after_a_sum():
    require_gpu()
    s, t = _solver(), _solver()
    for q in range(2):
        _add(s, q)
    x = rand_c((s.N, 8), 41)
    for precision in (0, 1, 2):
        s.interbody(x, precision=precision)
        s.interbody(np.ascontiguousarray(x[:, :1]), precision=precision)
    _add(s, 2)
    for q in range(3):
        _add(t, q)
    x = rand_c((t.N, 8), 42)
    assert s.N == t.N and np.array_equal(s.get_nodes()[0], t.get_nodes()[0])
    for precision, tol in ((0, 1e-13), (1, 1e-6), (2, 1e-12)):
        for cols in (8, 1):
            y = np.ascontiguousarray(x[:, :cols])
            got, want = s.interbody(y, precision=precision), t.interbody(y, precision=precision)
            assert np.abs(got - want).max() <= tol * np.abs(want).max(), (precision, cols)
