"""Workloads of exact N-Queens counting, through the package's public calls.

Every kind of call that a program makes is here: device-resident subproblems
(`nq.count`, `nq.count_ex`), whole boards (`nq.total`), few heavy host
subproblems (`nq.count_split`), partial-board queries (`nq.count_constrained`),
several boards replayed from one graph (`batch.Batch`) and a stream of requests
(`serve.Server`). Results are exact integers, so every tolerance is "exact".
"""
import math
import random
import time

import numpy as np
import torch

from paper_2511_12009_gb300 import batch, nq, serve

DEV = "cuda"


def listed():
    return [
        # A handful of small subtrees: the call's latency is all there is.
        {"name": "count_n10_d3", "kind": "count", "n": 10, "d": 3, "share": 0.9},
        # N = 14 in one launch from d = 3: about a thousand subtrees, far fewer
        # than the device has lanes.
        {"name": "count_n14_d3", "kind": "count", "n": 14, "d": 3, "share": 0.9},
        # N = 18 from d = 5: about 10^5 subtrees of uneven size, per-subtree counts.
        {"name": "count_n18_d5", "kind": "count", "n": 18, "d": 5, "share": 0.9},
        # N = 18 from d = 7: millions of subtrees already on the device (the
        # throughput workload; a worker's share of the canonical order).
        {"name": "count_n18_d7", "kind": "count", "n": 18, "d": 7, "share": 0.8},
        # A sample of N = 22 subtrees, as a long run spot-checks itself: few and heavy.
        {"name": "sample_n22_d7", "kind": "sample", "n": 22, "d": 7, "m": 2048},
        # Subproblems of several boards in one call, with weighted totals per board.
        {"name": "mixed_n12_17", "kind": "mixed", "lo": 12, "hi": 17, "d": 5, "m": 100003},
        # A table of Q(N) for small boards: latency of the whole-board call.
        {"name": "total_n4_11", "kind": "total", "lo": 4, "hi": 11},
        # The same for the boards that take the device tenths of a second.
        {"name": "total_n14_19", "kind": "total", "lo": 14, "hi": 19},
        # N = 27 subtrees on the host, fewer than there are lanes, each heavy.
        {"name": "split_n27_d10", "kind": "split", "n": 27, "d": 10, "m": 1024},
        # Partial boards: how many solutions hold the given queens.
        {"name": "constrained_n16", "kind": "constrained", "n": 16, "k": 2, "m": 6},
        # Five boards resident on the device, replayed as one graph.
        {"name": "batch_n13_17", "kind": "batch", "lo": 13, "hi": 17},
        # A burst of requests of several boards and constraints through the server.
        {"name": "serve_n10_15", "kind": "serve", "lo": 10, "hi": 15, "m": 32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count", "count", "count", "sample", "mixed", "total", "split",
                       "constrained", "batch", "serve"])
    if kind == "count":
        n = rng.randint(9, 18)
        return {"kind": kind, "n": n, "d": rng.randint(2, min(7, n - 4)),
                "share": round(rng.uniform(0.3, 0.95), 3)}
    if kind == "sample":  # at most 15 rows below the prefix, as at N = 22, d = 7
        n = rng.randint(17, 22)
        return {"kind": kind, "n": n, "d": n - rng.randint(10, 15), "m": _log_int(rng, 64, 4096)}
    if kind == "mixed":
        lo = rng.randint(8, 13)
        return {"kind": kind, "lo": lo, "hi": rng.randint(lo + 1, 17), "d": rng.randint(3, 6),
                "m": _log_int(rng, 1000, 200000)}
    if kind == "total":
        lo = rng.randint(1, 14)
        return {"kind": kind, "lo": lo, "hi": lo + 4}
    if kind == "split":
        n = rng.randint(22, 28)
        return {"kind": kind, "n": n, "d": n - rng.randint(13, 16), "m": _log_int(rng, 64, 2048)}
    if kind == "constrained":
        return {"kind": kind, "n": rng.randint(9, 17), "k": rng.randint(1, 4),
                "m": rng.randint(4, 8)}
    if kind == "batch":
        lo = rng.randint(6, 12)
        return {"kind": kind, "lo": lo, "hi": lo + 4}
    lo = rng.randint(8, 12)
    return {"kind": kind, "lo": lo, "hi": rng.randint(lo + 1, 15), "m": rng.randint(8, 48)}


# --- inputs ------------------------------------------------------------------

def _walks(rng, n, d, m, half=False):
    """m random placements of non-attacking queens in rows 0..d-1 (each row's
    column uniform among the free ones; a placement that gets stuck is drawn
    again): columns used, diagonals entering row d."""
    last = (1 << n) - 1
    out = np.zeros((0, 3), dtype=np.uint32)
    while len(out) < m:
        k = 2 * m + 64
        c, l, r = (np.zeros(k, dtype=np.int64) for _ in range(3))
        ok = np.ones(k, dtype=bool)
        for row in range(d):
            av = ~(c | l | r) & last
            if row == 0 and half:
                av &= (1 << (n // 2)) - 1
            bits = (av[:, None] >> np.arange(n)) & 1
            cnt = bits.sum(1)
            ok &= cnt > 0
            pick = (rng.random(k) * np.maximum(cnt, 1)).astype(np.int64)
            col = (bits.cumsum(1) <= pick[:, None]).sum(1)
            p = np.where(ok, np.int64(1) << np.minimum(col, n - 1), 0)
            c, l, r = c | p, ((l | p) << 1) & last, (r | p) >> 1
        out = np.concatenate([out, np.stack([c, l, r], 1)[ok].astype(np.uint32)])
    return out[:m]


def _records(state, n, d, weight=2):
    pre = np.zeros(len(state), dtype=nq.PREFIX_DTYPE)
    pre["cols"], pre["ld"], pre["rd"] = state[:, 0], state[:, 1], state[:, 2]
    pre["meta"] = weight | (n << 2) | (d << 7)
    return pre


def _queens(rng, n, k):
    """k queens on an n x n board, no two attacking each other."""
    while True:
        qs = []
        for _ in range(k):
            a = (rng.randrange(n), rng.randrange(n))
            if any(a[0] == b[0] or a[1] == b[1] or abs(a[0] - b[0]) == abs(a[1] - b[1])
                   for b in qs):
                break
            qs.append(a)
        if len(qs) == k:
            return qs


def _host_records(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "count":  # a worker's contiguous share of the canonical order
        pre = nq.enumerate_prefixes(case["n"], case["d"])
        m = max(1, int(len(pre) * case["share"]))
        first = int(rng.integers(0, len(pre) - m + 1))
        return pre[first:first + m]
    if kind in ("sample", "split"):
        return _records(_walks(rng, case["n"], case["d"], case["m"], True), case["n"], case["d"])
    # "mixed": boards lo..hi in any order, small boards' prefixes kept 3 rows above the end
    ns = rng.integers(case["lo"], case["hi"] + 1, case["m"])
    pre = np.zeros(case["m"], dtype=nq.PREFIX_DTYPE)
    for n in range(case["lo"], case["hi"] + 1):
        at = np.flatnonzero(ns == n)
        d = min(case["d"], n - 3)
        if len(at):
            pre[at] = _records(_walks(rng, n, d, len(at)), n, d, 1 + n % 2)
    return pre


_server = None


def _serve():
    """The program's one server, kept for its life (it leaves the GPU soon after a burst)."""
    global _server
    if _server is None:
        _server = serve.Server(max_n=20, request_slots=64, ring_records=1 << 22, idle_ms=1)
    return _server


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    rng = random.Random(seed)
    if kind in ("count", "sample", "mixed"):
        pre = _host_records(case, seed)
        s["pre"] = nq.to_device(pre, DEV)
        s["counts"] = torch.zeros(len(pre), dtype=torch.int64, device=DEV)
        if kind == "mixed":
            s["totals"] = torch.zeros(32, dtype=torch.int64, device=DEV)
            s["min_d"] = int(((pre["meta"] >> 7) & 31).min())
    elif kind == "split":
        s["pre"] = _host_records(case, seed)
    elif kind in ("total", "batch"):
        s["ns"] = list(range(case["lo"], case["hi"] + 1))
        rng.shuffle(s["ns"])  # the boards in the order that the program lists them
        if kind == "batch":
            s["batch"] = batch.Batch(s["ns"])
    elif kind == "constrained":
        s["queries"] = [_queens(rng, case["n"], case["k"]) for _ in range(case["m"])]
    else:
        s["server"] = _serve()
        s["requests"] = []
        for _ in range(case["m"]):
            n = rng.randint(case["lo"], case["hi"])
            s["requests"].append((n, _queens(rng, n, rng.randint(0, 4))))
    return s


def run(s):
    kind = s["kind"]
    if kind in ("count", "sample"):
        nq.count(s["n"], s["d"], s["pre"], s["counts"])
        return s["counts"]
    if kind == "mixed":
        s["totals"].zero_()
        nq.count_ex(s["pre"], s["min_d"], s["hi"], s["counts"], None, s["totals"])
        return [s["counts"], s["totals"]]
    if kind == "total":
        return [nq.total(n) for n in s["ns"]]
    if kind == "split":
        r = nq.count_split(s["pre"])
        return [r["counts"], r["totals"]]
    if kind == "constrained":
        return [nq.count_constrained(s["n"], q) for q in s["queries"]]
    if kind == "batch":
        return s["batch"].run()[0]
    srv, asked, answers = s["server"], {}, {}
    todo = list(enumerate(s["requests"]))
    while todo or asked:
        while todo:
            i, (n, q) = todo[0]
            t = srv.submit(n, q)
            if t is None:
                break
            asked[t] = i
            todo.pop(0)
        for t, count in srv.poll():
            answers[asked.pop(t)] = count
        if asked:
            time.sleep(20e-6)
    return np.array([answers[i] for i in range(len(answers))], dtype=np.int64)


# --- what a pass cannot do without -------------------------------------------

def _tree(n, d, given=False):
    """(prefixes of depth d in the half-symmetric set, queen placements below
    depth d), by Knuth's random-descent estimate with fixed draws; given: the
    placements below one prefix of depth d drawn by a random walk."""
    rng, k, last = np.random.default_rng(5), 20000, (1 << n) - 1
    c, l, r = (np.zeros(k, dtype=np.int64) for _ in range(3))
    w = np.ones(k)
    at_d, below = float(k), 0.0
    for row in range(n):
        av = ~(c | l | r) & last
        if row == 0:
            av &= (1 << ((n + 1) // 2)) - 1
        bits = (av[:, None] >> np.arange(n)) & 1
        cnt = bits.sum(1)
        if given and row == d:
            w = (w > 0).astype(float)
            k = max(1.0, w.sum())
        w = w * cnt
        if row + 1 == d:
            at_d = w.sum()
        if row >= d:
            below += w.sum()
        pick = (rng.random(len(c)) * np.maximum(cnt, 1)).astype(np.int64)
        col = np.minimum((bits.cumsum(1) <= pick[:, None]).sum(1), n - 1)
        p = np.where(cnt > 0, np.int64(1) << col, 0)
        c, l, r = c | p, ((l | p) << 1) & last, (r | p) >> 1
    return at_d / k, below / k


def _records_of(case):
    """(records, placements below them)."""
    kind = case["kind"]
    if kind == "count":
        at, below = _tree(case["n"], case["d"])
        return max(1.0, at * case["share"]), below * case["share"]
    if kind in ("sample", "split"):
        return case["m"], case["m"] * _tree(case["n"], case["d"], True)[1]
    boards = range(case["lo"], case["hi"] + 1)
    each = case["m"] / len(boards)
    return case["m"], sum(each * _tree(n, min(case["d"], n - 3), True)[1] for n in boards)


def work(case):
    """Bytes: each record once in, each count once out. Operations: ten 32-bit
    integer operations per queen placement below the given rows (lowest free
    column: 2, clear it, the three masks: 5, the next row's free columns: 2)."""
    kind = case["kind"]
    if kind in ("count", "sample", "mixed", "split"):
        m, nodes = _records_of(case)
        return {"bytes": 24 * m, "flops": 10 * nodes}
    if kind in ("total", "batch"):
        boards = range(case["lo"], case["hi"] + 1)
        return {"bytes": 8 * len(boards), "flops": 10 * sum(_tree(n, 0)[1] for n in boards)}
    if kind == "constrained":
        # a given queen takes its row and column and about 2(n-k) cells of the rest
        nodes = 2 * _tree(max(4, case["n"] - case["k"] - case["k"] // 2), 0)[1]
        return {"bytes": 8 * case["m"], "flops": 10 * case["m"] * nodes}
    boards = range(case["lo"], case["hi"] + 1)
    each = case["m"] / len(boards)
    nodes = sum(each * 0.4 * _tree(n, 0)[1] for n in boards)
    return {"bytes": 8 * case["m"], "flops": 10 * nodes}


def tolerance(case):
    return "exact"


# --- the same answers in plain numpy -------------------------------------------

def _below(c, l, r, n, rows, allowed=None, seg=None, nseg=0):
    """Completions of the states (c, l, r) at row n - rows, per segment."""
    last = np.int64((1 << n) - 1)
    for row in range(n - rows, n):
        av = ~(c | l | r) & last
        if allowed is not None:
            av &= allowed[row]
        src, bit = [], []
        for col in range(n):
            at = np.flatnonzero((av >> col) & 1)
            src.append(at)
            bit.append(np.full(len(at), np.int64(1) << col))
        src, p = np.concatenate(src), np.concatenate(bit)
        c, l, r = c[src] | p, ((l[src] | p) << 1) & last, (r[src] | p) >> 1
        seg = seg[src]
    return np.bincount(seg, minlength=nseg).astype(np.int64)


def _board(n, queens=()):
    """Solutions of the n x n board that contain every given queen."""
    allowed = [(1 << n) - 1] * n
    for r0, c0 in queens:
        for r in range(n):
            for c in range(n):
                if r == r0 and c != c0 or r != r0 and (c == c0 or abs(r - r0) == abs(c - c0)):
                    allowed[r] &= ~(1 << c)
    z = np.zeros(1, dtype=np.int64)
    return int(_below(z, z, z, n, n, allowed, z, 1)[0])


def exact(case, seed):
    """A breadth-first count in 64-bit numpy, for the sizes that it is quick at."""
    kind = case["kind"]
    if kind in ("total", "batch"):
        if case["hi"] > 11:
            return None
        ns = list(range(case["lo"], case["hi"] + 1))
        random.Random(seed).shuffle(ns)
        return [_board(n) for n in ns]
    if kind == "constrained":
        if case["n"] > 11:
            return None
        rng = random.Random(seed)
        return [_board(case["n"], _queens(rng, case["n"], case["k"])) for _ in range(case["m"])]
    if kind == "serve":
        if case["hi"] > 11:
            return None
        rng, out = random.Random(seed), []
        for _ in range(case["m"]):
            n = rng.randint(case["lo"], case["hi"])
            out.append(_board(n, _queens(rng, n, rng.randint(0, 4))))
        return np.array(out, dtype=np.int64)
    if case.get("hi", case.get("n")) > 11:
        return None
    pre = _host_records(case, seed)
    counts = np.zeros(len(pre), dtype=np.int64)
    totals = np.zeros(32, dtype=np.int64)
    ns, ds = (pre["meta"] >> 2) & 31, (pre["meta"] >> 7) & 31
    for n, d in sorted(set(zip(ns.tolist(), ds.tolist()))):
        at = np.flatnonzero((ns == n) & (ds == d))
        c, l, r = (pre[f][at].astype(np.int64) for f in ("cols", "ld", "rd"))
        counts[at] = _below(c, l, r, n, n - d, None, np.arange(len(at)), len(at))
        totals[n] += int((counts[at] * (pre["meta"][at] & 3)).sum())
    if kind == "count" or kind == "sample":
        return counts
    return [counts if kind == "mixed" else counts.astype(np.uint64), totals]
