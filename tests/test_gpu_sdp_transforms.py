"""Windows of the (+) recurrence by transforms: the edges of the range of a_1
that takes them, whole and halved chunks, a short last chunk, a window clipped
at the end of the table, and words that make every sum as large as it can be."""
import ctypes

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("amax", [2048, 2049, 2050, 4095, 4097, 8191, 8192, 8193])
@pytest.mark.parametrize("rows,chunks", [
    (9, 2), (9, 4),    # chunks of two or four windows: one factor of each kind
    (47, 11),          # chunks of four windows and a little
    (200, 3),          # halved chunks, P2 = 2
    (317, 30),         # halved, a remainder in both directions
    (640, 76), (640, 77),  # halved up to half a chunk per SM
])
@pytest.mark.parametrize("kind", ["random", "ones"])
def test_edges(amax, rows, chunks, kind):
    import torch
    import paper_2008_01938_gb300 as dp
    from paper_2008_01938_gb300 import native
    lib = native.load()
    r = np.random.RandomState(amax + rows)
    a = np.array([amax, amax - 1, 2000, 1177, 1031], dtype=np.int32)
    n = rows * amax + amax // 3 + 1
    preset = np.full(amax, 0xFFFFFFFF, np.uint32)
    if kind == "random":
        preset = r.randint(0, 1 << 32, amax, dtype=np.uint64).astype(np.uint32)
    st = np.zeros(n + 8, np.uint32)  # the words behind the table stay as they are
    st[:amax] = preset
    st[n:] = 0x5A5A5A5A
    t = torch.from_numpy(st.view(np.int32)).cuda()
    native.check(lib.dp_test_sdp_jump(ctypes.c_void_p(t.data_ptr()), n, ctypes.c_void_p(a.ctypes.data),
                                      int(a.size), chunks, None, None))
    dp.sync_status()
    got = t.cpu().numpy().view(np.uint32)
    bad = np.flatnonzero(got[:n] != oracle.sdp(preset, n, a, "add"))
    assert bad.size == 0, f"{bad.size} cells differ, first {bad[:5].tolist()}"
    assert (got[n:] == 0x5A5A5A5A).all()
