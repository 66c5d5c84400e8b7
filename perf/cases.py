"""The calls that a program using this package makes, as cases to be timed.

Every case goes through the package's public entry points.  Sizes are those of
the repository's own configurations, benchmark and tests: the 128- and
4096-matrix chains, the batch of uneven int64 chains, the 2^26-cell S-DP table,
the served request mix, and odd sizes between them.  All results are whole
numbers and are compared exactly.
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

import paper_2008_01938_gb300 as dp

DEV = "cuda"


def listed():
    return [
        # the smallest chain of the configurations, solved alone: latency and launches count
        {"name": "mcm_i32_128", "kind": "mcm", "n": 128, "cost": "i32", "dmax": 32},
        # the largest chain of the configurations: the headline solve
        {"name": "mcm_i32_4096", "kind": "mcm", "n": 4096, "cost": "i32", "dmax": 32},
        # one long chain with dims that need 64-bit costs, ragged last tile
        {"name": "mcm_i64_1500", "kind": "mcm", "n": 1500, "cost": "i64", "dmax": 1000},
        # a chain whose tables are wanted in page-locked host memory (wider dims: a smaller packing shift)
        {"name": "mcm_host_i32_1000", "kind": "mcm_host", "n": 1000, "cost": "i32", "dmax": 100},
        # thousands of uneven chains through one plan (dims of the batch configuration)
        {"name": "mcm_batch_i64_2000", "kind": "mcm_batch", "count": 2000, "nlo": 8, "nhi": 512, "cost": "i64",
         "dmax": 1000},
        # optimal binary search tree with 2000 gaps: the triangular DP with a weight per cell
        {"name": "interval_2000", "kind": "interval", "n": 2000, "fmax": 4},
        # the bracketing of a solved 4096-matrix chain
        {"name": "traceback_4096", "kind": "traceback", "n": 4096, "dmax": 32},
        # the 2^26-cell table of the configurations, both operators
        {"name": "sdp_min_2p26", "kind": "sdp", "op": "min", "n": 1 << 26, "k": 32, "amin": 1024, "amax": 8192,
         "ends": True},
        {"name": "sdp_add_2p26", "kind": "sdp", "op": "add", "n": 1 << 26, "k": 32, "amin": 1024, "amax": 8192,
         "ends": True},
        # a table of the served mix's lower range (odd length), summed
        {"name": "sdp_add_300k", "kind": "sdp", "op": "add", "n": 300001, "k": 16, "amin": 64, "amax": 4096,
         "ends": False},
        # many short tables through one plan
        {"name": "sdp_batch_min_200", "kind": "sdp_batch", "op": "min", "count": 200, "nlo": 1 << 12, "nhi": 1 << 16,
         "k": 16, "amin": 64, "amax": 4096},
        # a burst of the served mix: 80 % chains, 20 % tables, all submitted at once
        {"name": "serve_24", "kind": "serve", "count": 24, "mcm_nhi": 2048, "sdp_nhi": 1 << 22},
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(["mcm", "mcm", "mcm_host", "mcm_batch", "interval", "traceback", "sdp", "sdp", "sdp",
                       "sdp_batch", "serve"])
    if kind in ("mcm", "mcm_host"):
        cost = rng.choice(["i32", "i64"])
        n = _log_int(rng, 16, 2048 if cost == "i64" or kind == "mcm_host" else 4096)
        return {"kind": kind, "n": n, "cost": cost, "dmax": 1000 if cost == "i64" else rng.choice([32, 80])}
    if kind == "mcm_batch":
        cost = rng.choice(["i32", "i64"])
        return {"kind": kind, "count": _log_int(rng, 100, 2000), "nlo": rng.randint(1, 16),
                "nhi": _log_int(rng, 64, 512), "cost": cost, "dmax": 1000 if cost == "i64" else 100}
    if kind == "interval":
        return {"kind": kind, "n": _log_int(rng, 64, 2000), "fmax": rng.choice([4, 9, 100])}
    if kind == "traceback":
        return {"kind": kind, "n": _log_int(rng, 64, 4096), "dmax": 32}
    if kind == "sdp":
        amin = _log_int(rng, 1, 1024)
        amax = max(2 * amin + 64, _log_int(rng, 128, 8192))
        k = min(rng.choice([2, 4, 8, 16, 32, 48]), amin + 1)
        n = _log_int(rng, 1 << 14, min(1 << 26, amin << 15))
        return {"kind": kind, "op": rng.choice(["min", "add"]), "n": n, "k": k, "amin": amin, "amax": amax,
                "ends": rng.random() < 0.5}
    if kind == "sdp_batch":
        return {"kind": kind, "op": rng.choice(["min", "add"]), "count": _log_int(rng, 16, 400), "nlo": 1 << 12,
                "nhi": _log_int(rng, 1 << 13, 1 << 16), "k": rng.choice([4, 16, 32]), "amin": 64,
                "amax": rng.choice([1024, 4096])}
    return {"kind": "serve", "count": rng.randint(4, 24), "mcm_nhi": _log_int(rng, 256, 2048),
            "sdp_nhi": _log_int(rng, 1 << 17, 1 << 22)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _dims(r, n, dmax):
    return r.randint(1, dmax + 1, n + 1).astype(np.int32)


def _offsets(r, k, amin, amax, ends):
    """k distinct offsets in [amin, amax], descending; `ends` puts both limits among them."""
    if ends:
        mid = r.choice(np.arange(amin + 1, amax), k - 2, replace=False) if k > 2 else np.zeros(0, np.int64)
        a = np.concatenate([mid, [amin, amax]])
    else:
        a = r.choice(np.arange(amin, amax + 1), k, replace=False)
    return np.sort(a)[::-1].astype(np.int32).copy()


def _words(r, count):
    return r.randint(0, 1 << 32, count, dtype=np.uint64).astype(np.uint32)


def _log_sizes(count, lo, hi):
    """Log-uniform sizes; they belong to the case, so that the outputs of every seed have the same shapes."""
    r = np.random.RandomState(count)
    return np.minimum(hi, np.exp(r.uniform(math.log(lo), math.log(hi + 1), count)).astype(np.int64))


def _table(n, preset):
    st = torch.zeros(n, dtype=torch.int32, device=DEV)
    m = min(n, preset.size)
    st[:m] = torch.from_numpy(preset[:m].view(np.int32)).to(DEV)
    return st


def _requests(case, r):
    """The served mix: one table for every four chains, sizes log-uniform."""
    reqs, count = [], case["count"]
    chains, tables = _log_sizes(count, 16, case["mcm_nhi"]), _log_sizes(count, 1 << 16, case["sdp_nhi"])
    for i in range(count):
        if i % 5 != 4:
            n = int(chains[i])
            reqs.append({"kind": "mcm", "n": n, "dims": _dims(r, n, 1000)})
        else:
            n = int(tables[i])
            a = _offsets(r, 16, 64, 4096, False)
            reqs.append({"kind": "sdp", "n": n, "offs": a, "preset": _words(r, int(a[0]))})
    return reqs


def _weights(case, r):
    """Optimal-BST weights over n gaps: key and gap frequencies of each cell's range."""
    n, fmax = case["n"], case["fmax"]
    key = np.concatenate([[0], r.randint(1, fmax + 1, n - 1)])
    gap = r.randint(0, fmax + 1, n)
    kc = np.cumsum(key)
    gc = np.concatenate([[0], np.cumsum(gap)])
    kc, gc = torch.from_numpy(kc).to(DEV), torch.from_numpy(gc).to(DEV)
    w = (kc[None, :] - kc[:, None]) + (gc[None, 1:] - gc[:n, None])
    return torch.triu(w, 1).to(torch.int32).contiguous()


def _inputs(case, seed):
    """Everything that is drawn, in one order, for prepare() and exact()."""
    r = np.random.RandomState(seed % (1 << 32))
    kind = case["kind"]
    if kind in ("mcm", "mcm_host", "traceback"):
        return {"p": _dims(r, case["n"], case["dmax"])}
    if kind == "mcm_batch":
        ns = _log_sizes(case["count"], case["nlo"], case["nhi"]).astype(np.int32)
        return {"ns": ns, "p": r.randint(1, case["dmax"] + 1, int(ns.sum()) + ns.size).astype(np.int32)}
    if kind == "interval":
        return {"w": _weights(case, r)}
    if kind == "sdp":
        a = _offsets(r, case["k"], case["amin"], case["amax"], case["ends"])
        return {"offs": a, "preset": _words(r, int(a[0]))}
    if kind == "sdp_batch":
        ns = _log_sizes(case["count"], case["nlo"], case["nhi"])
        offs = [_offsets(r, case["k"], case["amin"], case["amax"], False) for _ in ns]
        return {"ns": ns, "offs": offs, "presets": [_words(r, int(a[0])) for a in offs]}
    return {"reqs": _requests(case, r)}


def prepare(case, seed):
    x = _inputs(case, seed)
    kind, st = case["kind"], {"case": case}
    if kind == "mcm":
        st["p"] = torch.from_numpy(x["p"]).to(DEV)
    elif kind == "mcm_host":
        n = case["n"]
        st["p"] = torch.from_numpy(x["p"]).pin_memory()
        dt = torch.int32 if case["cost"] == "i32" else torch.int64
        st["m"] = torch.empty((n, n), dtype=dt).pin_memory()
        st["s"] = torch.empty((n, n), dtype=torch.int16).pin_memory()
    elif kind == "mcm_batch":
        ns = x["ns"].astype(np.int64)
        p_off = np.concatenate([[0], np.cumsum(ns + 1)])
        t_off = np.concatenate([[0], np.cumsum(ns * ns)])
        st["plan"] = dp.McmPlan(x["ns"], cost=case["cost"])
        st["p"] = torch.from_numpy(x["p"]).to(DEV)
        st["p_off"] = torch.from_numpy(p_off[:-1].copy()).to(DEV)
        st["t_off"] = torch.from_numpy(t_off[:-1].copy()).to(DEV)
        dt = torch.int32 if case["cost"] == "i32" else torch.int64
        st["m"] = torch.empty(int(t_off[-1]), dtype=dt, device=DEV)
        st["s"] = torch.empty(int(t_off[-1]), dtype=torch.int16, device=DEV)
    elif kind == "interval":
        st["p"] = torch.zeros(case["n"] + 1, dtype=torch.int32, device=DEV)
        st["w"] = x["w"]
    elif kind == "traceback":
        st["s"] = dp.mcm_solve(torch.from_numpy(x["p"]).to(DEV))[1]
    elif kind == "sdp":
        st["offs"] = x["offs"]
        st["st"] = _table(case["n"], x["preset"])
    elif kind == "sdp_batch":
        sizes = [max(int(n), int(a[0])) for n, a in zip(x["ns"], x["offs"])]
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        tab = np.zeros(int(off[-1]), np.uint32)
        for o, pre in zip(off, x["presets"]):
            tab[o:o + pre.size] = pre
        st["plan"] = dp.SdpPlan(x["ns"], x["offs"], op=case["op"])
        st["st"] = torch.from_numpy(tab.view(np.int32)).to(DEV)
        st["off"] = torch.from_numpy(off[:-1].copy()).to(DEV)
    else:
        st["reqs"] = x["reqs"]
        st["srv"] = dp.Server(hbm_cap_bytes=16 << 30, max_inflight=1024)
        st["out"] = [
            (torch.empty((q["n"], q["n"]), dtype=torch.int64, device=DEV),
             torch.empty((q["n"], q["n"]), dtype=torch.int16, device=DEV)) if q["kind"] == "mcm"
            else torch.empty(q["n"], dtype=torch.int32, device=DEV) for q in x["reqs"]]
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _serve(st):
    """Submits the burst, takes each result into the program's own buffers as it finishes, and releases it."""
    srv, waiting = st["srv"], {}
    for i, q in enumerate(st["reqs"]):
        t = srv.submit_mcm(q["dims"]) if q["kind"] == "mcm" else srv.submit_sdp(q["n"], q["offs"], q["preset"])
        if t is None:
            raise RuntimeError("the server refused a request")
        waiting[t] = i
    end = time.monotonic() + 30
    while waiting:
        for t in list(waiting):
            res = srv.poll(t)
            if res is None:
                continue
            if res.status != 0:
                raise RuntimeError("a request ended with status %d" % res.status)
            got, own = srv.tables(res), st["out"][waiting.pop(t)]
            if isinstance(own, tuple):
                own[0].copy_(got[0])
                own[1].copy_(got[1])
            else:
                own.copy_(got)
            srv.release(t)
        if time.monotonic() > end:
            raise RuntimeError("the server did not finish")
    return st["out"]


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "mcm":
        return dp.mcm_solve(state["p"], cost=c["cost"])
    if kind == "mcm_host":
        return dp.mcm_solve_host(state["p"], cost=c["cost"], m=state["m"], s=state["s"])
    if kind == "mcm_batch":
        state["plan"].solve(state["p"], state["p_off"], state["t_off"], state["m"], state["s"])
        return state["m"], state["s"]
    if kind == "interval":
        return dp.interval_dp_solve(state["p"], state["w"])
    if kind == "traceback":
        return dp.mcm_traceback(state["s"])
    if kind == "sdp":
        return dp.sdp_solve(state["st"], state["offs"], op=c["op"])
    if kind == "sdp_batch":
        state["plan"].solve(state["st"], state["off"])
        return state["st"]
    return _serve(state)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _log_mean(f, lo, hi):
    """The mean of f(n) for n log-uniform in [lo, hi]."""
    x = np.exp(np.linspace(math.log(lo), math.log(hi + 1), 257))
    return float(np.mean(f(x)))


def _mcm_work(n, es, extra=0):
    """Tables written once (and `extra` bytes a cell above the diagonal read once); a multiply-add, an add and a
    minimum per split."""
    return np.array([n * n * (es + 2) + 4 * n + extra * n * n / 2, 3 * (n ** 3 - n) / 6])


def work(case):
    kind = case["kind"]
    es = 8 if case.get("cost") == "i64" else 4
    if kind in ("mcm", "mcm_host"):
        w = _mcm_work(case["n"], es)
    elif kind == "mcm_batch":
        w = case["count"] * np.array([_log_mean(lambda n, i=i: _mcm_work(n, es)[i], case["nlo"], case["nhi"])
                                      for i in (0, 1)])
    elif kind == "interval":
        w = _mcm_work(case["n"], 4, 4)
    elif kind == "traceback":
        w = np.array([case["n"] * (2 + 12), case["n"]])
    elif kind == "sdp":  # the preset is read, the other cells are written; one combination per cell at least
        w = np.array([4 * case["n"], case["n"]])
    elif kind == "sdp_batch":
        w = case["count"] * _log_mean(lambda n: n, case["nlo"], case["nhi"]) * np.array([4, 1])
    else:  # solved, and copied out
        mcm, sdp = case["count"] - case["count"] // 5, case["count"] // 5
        w = mcm * np.array([_log_mean(lambda n, i=i: _mcm_work(n, 8)[i], 16, case["mcm_nhi"]) for i in (0, 1)])
        w = w + sdp * _log_mean(lambda n: n, 1 << 16, case["sdp_nhi"]) * np.array([4, 1])
        w = w + np.array([2 * w[0], 0])
    return {"bytes": float(w[0]), "flops": float(w[1])}


def tolerance(case):
    return "exact"  # whole numbers, wrapping sums included


# ---------------------------------------------------------------------------
# the same results by plain torch, in 64 bits
# ---------------------------------------------------------------------------

def _exact_chain(p, w=None):
    """m and s of the chain, diagonal by diagonal."""
    n = int(p.numel()) - 1
    p = p.to(DEV, torch.int64)
    by_start = torch.zeros((n, n), dtype=torch.int64, device=DEV)  # [d][i] = m[i][i + d]
    by_end = torch.zeros((n, n), dtype=torch.int64, device=DEV)    # [d][j] = m[j - d][j]
    m = torch.zeros((n, n), dtype=torch.int64, device=DEV)
    s = torch.full((n, n), -1, dtype=torch.int64, device=DEV)
    i = torch.arange(n, device=DEV)
    for d in range(1, n):
        a = i[:n - d]
        t = i[:d, None]
        cand = by_start[:d, :n - d] + by_end[:d, d:].flip(0)
        cand += p[:n - d][None, :] * p[a[None, :] + t + 1] * p[d + 1:][None, :]
        best = cand.min(0).values
        first = torch.where(cand == best, t, d).min(0).values
        v = best if w is None else best + w[a, a + d]
        by_start[d, :n - d] = v
        by_end[d, d:] = v
        m[a, a + d] = v
        s[a, a + d] = a + first
    return m, s


def _exact_table(n, offs, preset, op):
    """The table, as many cells at a time as the smallest offset."""
    st = torch.zeros(max(n, preset.size), dtype=torch.int64, device=DEV)
    st[:preset.size] = torch.from_numpy(preset.astype(np.int64)).to(DEV)
    a = torch.from_numpy(offs.astype(np.int64)).to(DEV)
    step = int(offs[-1])
    rows = torch.arange(step, device=DEV)[:, None] - a[None, :]
    for at in range(int(offs[0]), n, step):
        c = min(step, n - at)
        v = st[rows[:c] + at]
        st[at:at + c] = v.min(1).values if op == "min" else v.sum(1) & 0xFFFFFFFF
    return st


def _wrapped(st):
    return torch.where(st >= 1 << 31, st - (1 << 32), st).to(torch.int32)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("mcm_batch", "sdp_batch"):
        return None  # hundreds of thousands of small steps: longer than 20 seconds
    x = _inputs(case, seed)
    if kind in ("mcm", "mcm_host"):
        m, s = _exact_chain(torch.from_numpy(x["p"]))
        return m.to(torch.int32 if case["cost"] == "i32" else torch.int64), s.to(torch.int16)
    if kind == "interval":
        n = case["n"]
        m, s = _exact_chain(torch.zeros(n + 1, dtype=torch.int64), x["w"].to(torch.int64))
        return m.to(torch.int32), s.to(torch.int16)
    if kind == "traceback":
        s = _exact_chain(torch.from_numpy(x["p"]))[1].cpu().numpy()
        steps, stack = [], [(0, case["n"] - 1)]
        while stack:  # root, right, left: the reverse of post-order
            i, j = stack.pop()
            if i < j:
                k = int(s[i, j])
                steps.append((i, k, j))
                stack += [(i, k), (k + 1, j)]
        return torch.tensor(steps[::-1], dtype=torch.int32)
    if kind == "sdp":
        if (case["n"] - int(x["offs"][0])) // int(x["offs"][-1]) > 200000:
            return None
        return _wrapped(_exact_table(case["n"], x["offs"], x["preset"], case["op"])[:case["n"]])
    out = []
    for q in x["reqs"]:
        if q["kind"] == "mcm":
            m, s = _exact_chain(torch.from_numpy(q["dims"]))
            out.append((m, s.to(torch.int16)))
        else:
            out.append(_wrapped(_exact_table(q["n"], q["offs"], q["preset"], "min")[:q["n"]]))
    return out
