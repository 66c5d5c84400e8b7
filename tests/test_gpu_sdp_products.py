"""The products modulo the characteristic polynomial at the edges of their
blocks: one split piece and several, an output block filled to its last word,
levels of few and of many products."""
import ctypes

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("amax", [2, 3, 127, 128, 129, 1920, 1921, 1922, 2047, 2048, 9001])
@pytest.mark.parametrize("chunks", [2, 13, 152])
@pytest.mark.parametrize("rows", [3, 41])
def test_edges(amax, chunks, rows):
    import torch
    import paper_2008_01938_gb300 as dp
    from paper_2008_01938_gb300 import native
    lib = native.load()
    r = np.random.RandomState(amax + chunks)
    a = np.unique(np.r_[amax, max(1, amax - 1), max(1, amax // 2), max(1, amax // 7)])[::-1].astype(np.int32).copy()
    n = rows * chunks * amax + amax // 2 + 1
    preset = r.randint(0, 1 << 32, amax, dtype=np.uint64).astype(np.uint32)
    st = np.zeros(n, np.uint32)
    st[:amax] = preset
    t = torch.from_numpy(st.view(np.int32)).cuda()
    native.check(lib.dp_test_sdp_jump(ctypes.c_void_p(t.data_ptr()), n, ctypes.c_void_p(a.ctypes.data),
                                      int(a.size), chunks, None, None))
    dp.sync_status()
    bad = np.flatnonzero(t.cpu().numpy().view(np.uint32) != oracle.sdp(preset, n, a, "add"))
    assert bad.size == 0, f"{bad.size} cells differ, first {bad[:5].tolist()}"
