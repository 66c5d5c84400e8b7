"""(+) requests served together: those solved in chunks, those that share a
launch, and short and preset-only ones, in groups that split either way."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [
    [200000],                                  # alone: in chunks
    [200000] * 12,                             # as many launches would take longer: one launch
    [1 << 22, 200000, 200000, 150000, 90000],  # the long one in chunks, the others together
    [1 << 22, 1 << 21, 3000, 900, 1000],       # two in chunks; short and preset-only ones
])
def test_groups(lengths):
    import paper_2008_01938_gb300 as dp
    r = np.random.RandomState(len(lengths))
    a = np.sort(np.r_[64, 1000, r.choice(np.arange(65, 1000), 14, replace=False)])[::-1].astype(np.int32)
    presets = [r.randint(0, 1 << 32, 1000, dtype=np.uint64).astype(np.uint32) for _ in lengths]
    srv = dp.Server()
    tickets = [srv.submit_sdp(n, a, p, op="add") for n, p in zip(lengths, presets)]
    for n, p, t in zip(lengths, presets, tickets):
        while (res := srv.poll(t)) is None:
            pass
        got = srv.tables(res)
        got = (got[0] if isinstance(got, tuple) else got).cpu().numpy().view(np.uint32)[:n]
        assert np.array_equal(got, oracle.sdp(p, n, a, "add")[:n])
        srv.release(t)
    srv.close()


@pytest.mark.parametrize("op", ["min", "add"])
@pytest.mark.parametrize("others", [[], [200000, 1 << 22], [200000] * 6 + [900, 1000]])
def test_a_wide_window_among_others(op, others):
    """A window too wide for the ring is solved beside the others of its group
    (first, last, and alone in the group)."""
    import paper_2008_01938_gb300 as dp
    r = np.random.RandomState(len(others))
    a = np.sort(np.r_[64, 1000, r.choice(np.arange(65, 1000), 14, replace=False)])[::-1].astype(np.int32)
    wide = np.array([40000, 39000, 1024], np.int32)
    requests = [(130001, wide)] + [(n, a) for n in others] + [(90000, wide), (40000, wide)]
    presets = [r.randint(0, 1 << 32, q[0], dtype=np.uint64).astype(np.uint32) for _, q in requests]
    srv = dp.Server()
    tickets = [srv.submit_sdp(n, q, p, op=op) for (n, q), p in zip(requests, presets)]
    for (n, q), p, t in zip(requests, presets, tickets):
        while (res := srv.poll(t)) is None:
            pass
        assert res.status == 0
        got = srv.tables(res).cpu().numpy().view(np.uint32)[:n]
        assert np.array_equal(got, oracle.sdp(p, n, q, op)[:n])
        srv.release(t)
    srv.close()
