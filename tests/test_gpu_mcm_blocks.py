"""The int32 in-tile solves (2x2-cell blocks; the triangle of a diagonal tile by
pairs of rows): lengths around the edges of blocks, pairs and tiles, many splits
of equal cost, and the interval DP's weights."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

NS = [2, 3, 15, 16, 17, 30, 31, 32, 33, 34, 35, 47, 48, 62, 63, 64, 65, 66, 96, 97, 127, 161, 290]


@pytest.mark.parametrize("n", NS)
@pytest.mark.parametrize("hi", [1, 3, 20, 80])
def test_mcm(n, hi):
    import torch
    import paper_2008_01938_gb300 as dp
    p = np.random.RandomState(n + hi).randint(1, hi + 1, n + 1).astype(np.int32)
    m, s = dp.mcm_solve(torch.from_numpy(p).cuda(), cost="i32")
    dp.sync_status()
    om, os_ = oracle.mcm(p)
    assert np.array_equal(m.cpu().numpy(), om) and np.array_equal(s.cpu().numpy(), os_)


@pytest.mark.parametrize("n", NS)
@pytest.mark.parametrize("phi,whi", [(1, 5), (6, 1), (8, 500)])
def test_interval(n, phi, whi):
    import torch
    import paper_2008_01938_gb300 as dp
    r = np.random.RandomState(n + phi + whi)
    p = r.randint(0, phi + 1, n + 1).astype(np.int32)
    w = np.triu(r.randint(0, whi + 1, (n, n)), 1).astype(np.int32)
    m, s = dp.interval_dp_solve(torch.from_numpy(p).cuda(), torch.from_numpy(w).cuda())
    dp.sync_status()
    om, os_ = oracle.interval(p, w)
    assert np.array_equal(m.cpu().numpy(), om) and np.array_equal(s.cpu().numpy(), os_)
