"""The periodic tail of a min S-DP table: where the host says it starts (CPU,
against the oracle's whole tables), and the tables the GPU writes there."""
import ctypes
import math
import random

import numpy as np
import pytest

import oracle
from paper_2008_01938_gb300 import native

# (offsets, n): gcd 1 with 1, 2 and many offsets, consecutive ones, a common
# factor (below and above 64, and a_1 itself), tables that end before or just
# after the tail starts, offsets inside one word, k above the register limit
CASES = [
    ([1], 40), ([2, 1], 300), ([7, 5], 200), ([64, 63], 9000), ([1055 - i for i in range(32)], 60000),
    ([96, 90, 84], 3000), ([130, 65], 2000), ([4096, 2048, 1024], 20000), ([500], 5001), ([900, 890, 700, 64], 9001),
    ([3000, 2999, 1], 30000), ([8192, 7000, 5001, 3333, 1024], 200003), ([61, 53, 50, 40, 33, 17, 9], 1111),
    ([2000 - 3 * i for i in range(48)], 40002), ([20000, 16000, 1500], 150000), ([40, 30], 111),
]


def tail(a, n):
    a = np.asarray(a, np.int32)
    g = ctypes.c_int32()
    t = native.load().dp_test_sdp_min_tail(n, ctypes.c_void_p(a.ctypes.data), int(a.size), ctypes.byref(g))
    return int(t), int(g.value)


def table(a, n, seed):
    preset = np.random.RandomState(seed).randint(0, 1 << 32, a[0], dtype=np.uint64).astype(np.uint32)
    return preset, oracle.sdp(preset, n, np.asarray(a, np.int32), "min")


@pytest.mark.parametrize("a,n", CASES)
def test_tail_repeats_the_class_minima(a, n):
    t, g = tail(a, n)
    assert 0 <= t < n
    if t == 0:
        return
    assert g == math.gcd(*a) and t > a[0]
    preset, ref = table(a, n, len(a))
    cls = np.array([preset[r::g].min() for r in range(g)], np.uint32)
    at = np.arange(t - g, n)
    assert np.array_equal(ref[t - g:], cls[at % g])


def test_tail_is_found_where_it_matters():
    assert tail([1055 - i for i in range(32)], 60000)[0] > 0
    assert tail([8192, 7000, 5001, 3333, 1024], 200003)[0] > 0
    assert tail([4096, 2048, 1024], 20000)[1] == 1024
    assert tail([8192, 8191], 1 << 26)[0] == 0  # fills in too slowly to be found


def random_offsets(r):
    hi = int(2 ** r.uniform(1, 8))
    lo = max(1, int(hi * r.choice([0.05, 0.3, 0.7, 0.9])))
    k = min(r.randint(1, 6), hi - lo + 1)
    return sorted((x * r.choice([1, 2, 3]) for x in r.sample(range(lo, hi + 1), k)), reverse=True)


@pytest.mark.parametrize("seed", range(4))
def test_tail_is_given_up_only_where_there_is_none(seed):
    """Against the sums themselves: the first of a_k / g consecutive ones says
    where the tail starts, and a table that reaches past them has one."""
    r = random.Random(seed)
    for _ in range(400):
        a = sorted(set(random_offsets(r)), reverse=True)
        g = math.gcd(*a)
        b = [x // g for x in a]
        top = 65 * max(b) + 64
        sums = 1
        for x in b:
            while (more := (sums | sums << x) & ((1 << top) - 1)) != sums:
                sums = more
        run = sums
        for i in range(1, b[-1]):
            run &= sums >> i
        c = (run & -run).bit_length() - 1
        if c < 0:
            continue
        gap = max(x - y for x, y in zip(a, a[1:] + [0]))
        start = g * c + a[0] - 1 + gap + g  # the tail
        for n in (start - 5, start):
            assert tail(a, n)[0] == 0, (a, n)
        for n in (start + a[-1] + 64 * g, 2 * start + a[-1] + 64 * g):  # (room for the whole run)
            assert tail(a, n)[0] == start, (a, n)


@pytest.mark.parametrize("n, a", [
    (1 << 20, [8192, 8191]),                    # sums of m offsets stay apart: nothing to search for
    (1 << 18, [4000, 3001]), (65536, [1200, 801]),
    (55786, [7935 - 46 * i for i in range(32)]),  # a short table of many offsets
    (76589, [23045 - 1239 * i for i in range(16)]), (97000, [9000, 8501, 8102, 7503]),
    (1 << 26, [16000, 9000, 7001]),
])
def test_search_is_small_beside_the_solve(n, a):
    """The host's search for a tail (1.2 word operations or more per ns) takes
    at most half of the time that the steps take."""
    a = np.asarray(a, np.int32)
    plain = ctypes.c_int64()
    ops = native.load().dp_test_sdp_min_tail_ops(n, ctypes.c_void_p(a.ctypes.data), int(a.size), ctypes.byref(plain))
    assert 0 <= ops <= max(0.5 * 1.2 * plain.value, a.size + 8)
    if a.size == 2:
        assert ops == 0


SPREAD = list(range(1000, 63, -67)) + [64]  # 16 offsets, window on chip
WIDE = [40000, 39000, 1024]                 # window too wide for the ring


def share(requests, op):
    """The server's decision for a group: (launch, whether the tail is written) per request."""
    n = np.array([r[0] for r in requests], np.int64)
    k = np.array([len(r[1]) for r in requests], np.int32)
    offs = np.concatenate([np.asarray(r[1], np.int32) for r in requests])
    out = np.zeros(n.size, np.int32)
    ptr = lambda x: ctypes.c_void_p(x.ctypes.data)  # noqa: E731
    assert native.load().dp_test_serve_sdp_share(n.size, ptr(n), ptr(k), ptr(offs), op, 152, ptr(out)) == n.size
    return [(("ring", "off ring", "own")[x & 255], bool(x & 256)) for x in out]


@pytest.mark.parametrize("op", [0, 1])
@pytest.mark.parametrize("others", [[200000], [200000] * 12, [1 << 22, 200000, 90000, 500]])
@pytest.mark.parametrize("wide", [300000, 1 << 22])
def test_a_wide_window_leaves_a_served_group_its_routes(op, others, wide):
    """A request whose window does not fit on chip goes off the ring by itself:
    the others are solved as they would be without it."""
    group = [(n, SPREAD) for n in others]
    alone = share(group, op)
    for at in (0, len(group)):
        got = share(group[:at] + [(wide, WIDE)] + group[at:], op)
        assert got.pop(at) == ("off ring", False)
        assert got == alone
    assert all(g[0] != "off ring" for g in alone)
    assert all(g[1] for g, n in zip(alone, others) if n > 10000) if op == 0 else not any(g[1] for g in alone)


@pytest.mark.gpu
@pytest.mark.parametrize("a,n", CASES + [([8192, 7000, 5001, 3333, 1024], 5000003), ([1280, 768, 256], 1 << 20)])
@pytest.mark.parametrize("shift", [0, 1])
def test_tail_on_the_gpu(a, n, shift):
    import torch
    import paper_2008_01938_gb300 as dp
    preset, ref = table(a, n, len(a) + 1)
    buf = torch.full((n + 8,), -7, dtype=torch.int32, device="cuda")  # `shift`: a table off the 16-byte boundary
    st = buf[shift:shift + n]
    st[:a[0]] = torch.from_numpy(preset.view(np.int32)).cuda()
    dp.sdp_solve(st, a, op="min")
    plan = dp.SdpPlan([n, n - 1], [a, a], op="min")
    both = torch.full((2 * n + 8,), -7, dtype=torch.int32, device="cuda")
    off = torch.tensor([shift, n + shift + 1], device="cuda")
    for o in (shift, n + shift + 1):
        both[o:o + a[0]] = torch.from_numpy(preset.view(np.int32)).cuda()
    plan.solve(both, off)
    dp.sync_status()
    assert np.array_equal(st.cpu().numpy().view(np.uint32), ref)
    assert torch.all(buf[:shift] == -7) and torch.all(buf[shift + n:] == -7)
    for o, c in ((shift, n), (n + shift + 1, n - 1)):
        assert np.array_equal(both[o:o + c].cpu().numpy().view(np.uint32), ref[:c])
    assert torch.all(both[n + shift:n + shift + 1] == -7) and torch.all(both[2 * n + shift:] == -7)
