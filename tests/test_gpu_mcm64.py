"""The int64-cost MCM kernel at the edges of its tiles, of its blocks of 8 cells
and of its segments, with ties, combs and costs next to the bound."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _dims(kind, n, r):
    if kind == "random":
        return r.randint(1, 1001, n + 1)
    if kind == "ties":            # few values: many splits of equal cost
        return r.randint(1, 4, n + 1)
    if kind == "equal":
        return np.full(n + 1, 7)
    if kind == "rising":
        return np.arange(1, n + 2)
    if kind == "valley":
        return np.abs(np.arange(n + 1) - n // 2) + 1
    c = int((2 ** 47 - 1) // max(n - 1, 1)) ** (1 / 3)  # the largest dims the bound allows
    return np.full(n + 1, max(1, min(65535, int(c) - 1)))


@pytest.mark.parametrize("kind", ["random", "ties", "equal", "rising", "valley", "bound"])
@pytest.mark.parametrize("n", [1, 2, 8, 9, 31, 32, 33, 40, 63, 64, 65, 72, 95, 97, 129, 161, 200, 259])
def test_edges(kind, n):
    import torch
    import paper_2008_01938_gb300 as dp
    p = _dims(kind, n, np.random.RandomState(n)).astype(np.int32)
    m, s = dp.mcm_solve(torch.from_numpy(p).cuda(), cost="i64")
    dp.sync_status()
    om, os_ = oracle.mcm(p)
    assert np.array_equal(m.cpu().numpy(), om) and np.array_equal(s.cpu().numpy(), os_)
