"""The step kernel's variants at their edges: offset counts around 4, 8, 16, 24
and 32, steps narrower and wider than a warp or a block, each kind of window."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 3, 4, 5, 8, 9, 12, 15, 16, 17, 24, 31, 32, 33, 40, 49])
@pytest.mark.parametrize("amin,amax", [(1, 200), (33, 3000), (257, 9000), (1024, 16500), (1500, 33000)])
def test_every_offset_count(k, amin, amax):
    import torch
    import paper_2008_01938_gb300 as dp
    r = np.random.RandomState(1000 * k + amin)
    a = np.sort(np.concatenate([[amin], r.choice(np.arange(amin + 1, amax), k - 1, replace=False)]))[::-1]
    short = a[: max(1, k - 3)]  # in the batch: fewer offsets than the widest instance
    n = int(a[0]) + 5 * amin + 77
    presets = [r.randint(0, 1 << 32, a[0], dtype=np.uint64).astype(np.uint32) for _ in range(3)]
    for op in ("min", "add"):
        st = np.zeros((3, n), np.uint32)
        for row, p in zip(st, presets):
            row[: p.size] = p
        t = torch.from_numpy(st.view(np.int32).copy()).cuda().reshape(-1)
        dp.sdp_solve(t[:n], a, op=op)
        plan = dp.SdpPlan([n, n - 3], [a, short], op=op)
        plan.solve(t, torch.tensor([n, 2 * n], device="cuda"))
        dp.sync_status()
        got = t.cpu().numpy().view(np.uint32).reshape(3, n)
        assert np.array_equal(got[0], oracle.sdp(presets[0], n, a.astype(np.int32), op))
        assert np.array_equal(got[1], oracle.sdp(presets[1], n, a.astype(np.int32), op))
        ref = oracle.sdp(presets[2][: short[0]], n - 3, short.astype(np.int32), op)
        assert np.array_equal(got[2][: n - 3], ref)
