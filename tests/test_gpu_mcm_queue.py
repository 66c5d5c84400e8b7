"""The work queue as the device builds it against the host's: the same tasks,
and the same kind of task at every place (the host's order is checked for its
dependencies on the CPU; tasks of one kind do not depend on each other)."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _queue(f, ns):
    a = np.asarray(ns, np.int32)
    p = ctypes.c_void_p(a.ctypes.data)
    count = f(p, a.size, 1, None, 0)
    out = np.zeros((count, 6), np.int32)
    assert f(p, a.size, 1, ctypes.c_void_p(out.ctypes.data), count) == count
    return out


@pytest.mark.parametrize("ns", [[1], [32], [33], [300], [1025], [4096], [7000], [1, 2, 31, 32, 33],
                                [512, 9, 400, 64, 65, 8, 300, 511] * 40, [2048, 17, 1999]])
def test_device_queue_matches_the_hosts(ns):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2008_01938_gb300 import native
    lib = native.load()
    host, dev = _queue(lib.dp_test_mcm_queue, ns), _queue(lib.dp_test_mcm_device_queue, ns)
    if len(ns) == 1:
        assert np.array_equal(host, dev)
    key = lambda q: np.stack([q[:, 3], q[:, 2] - q[:, 1], (q[:, 3] == 1) & (q[:, 5] == q[:, 2] - q[:, 1] - 2)], 1)
    assert np.array_equal(key(host), key(dev))  # kind, tile-diagonal, whether a last part
    order = lambda q: q[np.lexsort(q.T[::-1])]
    assert np.array_equal(order(host), order(dev))
