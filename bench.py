"""Benchmark: exact N-Queens counting on GB300 -- search nodes/s, solve time,
integer-roofline fraction.

One step = one pass of the whole device hot path over one batch: the persistent
search kernel over every subproblem of the N=18 board (per-prefix uint64 counts
written, weighted totals reduced per warp) with the prefixes already resident
in HBM. The end-to-end number (``e2e``) goes through the public C call
nq_total_ex: host enumeration, pinned host->device copy, search, device->host
read of the total, every step.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

Prints one JSON line (rank 0). ``--impl reference`` times the CPU oracle on
the host cores instead (a bounded sample per step).
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "search nodes/s and exact-count solve time at N=18/22 on 1 GB300; ALU roofline %"
UNIT = "nodes/s"
# 32-bit integer operations of the search per node (one queen placement):
# neg+and (lowest bit), xor (clear it), or (cols), or+shl (ld), or+shr (rd),
# nor3 (next row) -- the algorithmic work of Algorithm 2's loop body.
ALU_OPS_PER_NODE = 10
# The integer roofline. The search issues its 32-bit integer work on two pipes:
# the ALU pipe (logic, compares, selects, shifts: 64 lanes/clk/SM, measured by
# nq_probe_alu's lop3/shf rates) and the FMA pipe (the multiply-add form of the
# disjoint-bit arithmetic and the moves ptxas places there: another 64; the
# probe's add rate, 127 lanes/clk/SM, is both pipes together). Together they
# equal the issue rate, 4 warp schedulers x 32 lanes = 128 lanes/clk/SM: the
# peak integer-op rate of the SM for this instruction mix. The ALU pipe alone
# is kept beside it as a secondary figure.
INT_LANES_PER_CLK_SM = 128
ALU_PIPE_LANES_PER_CLK_SM = 64
SM_MAX_MHZ_FALLBACK = 2070.0
# Prefix depth of the library's default (nq_default_depth), restated here so
# that the reference arm does not load the library: 7 up to N = 22, else 6,
# never more than N - 2.
def default_depth(n: int) -> int:
    return max(0, min(7 if n <= 22 else 6, n - 2))


# Search nodes (queen placements in rows 7..21) below the 60,760,010 depth-7
# prefixes of N = 22, counted by the library's diagnostic kernel build (its
# per-prefix node counts equal the oracle's on the seeded N = 22 sample and on
# every prefix of N <= 19); `--n22-nodes` counts them again.
N22_D7_NODES = 143257329200995
# DRAM traffic of one production search launch on the default workload (N=18,
# d=7, default layout), dram__bytes_read.sum + dram__bytes_write.sum from one
# ncu capture, valid only for the sources it was taken on: the sha256 of
# KERNEL_FILES. Any change to them makes the figure stale, and the roofline then
# reports traffic as null.
TRAFFIC_NCU = {"n": 18, "d": 7, "layout": "default", "bytes": 119246080 + 29120256,
               "kernel_sha256": "647949bf5c835def50a0680cc72b5d2ae60a7cc2d17b6f05cf463c9206798f59"}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=18)
    ap.add_argument("--d", type=int, default=0, help="prefix depth (0 = library default)")
    ap.add_argument("--layout", default="default",
                    choices=["default", "paper", "reg", "wt", "wt32", "wt32a", "wtm", "regm",
                             "regp", "regz", "regpz", "avail"])
    ap.add_argument("--block", type=int, default=0)
    ap.add_argument("--bps", type=int, default=0, help="blocks per SM (0 = max)")
    ap.add_argument("--order", type=int, default=0, help="0 default, 1 index order, 2 reverse")
    ap.add_argument("--e2e-steps", type=int, default=5)
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--workload", default="n18", choices=["n18", "batched", "served", "probe27"],
                    help="n18: the full N (default 18) count; batched: N=16..21 in one graph "
                         "launch vs one launch each; served: Poisson request stream; "
                         "probe27: 4096 seeded N=27 subtrees")
    ap.add_argument("--no-n22", action="store_true", help="skip the N=22 solve")
    ap.add_argument("--no-extras", action="store_true",
                    help="skip the short N=14, batched and served measurements of the default line")
    ap.add_argument("--n22-nodes", action="store_true",
                    help="count the N=22 nodes with the diagnostic build (about 2.5 min)")
    ap.add_argument("--requests", type=int, default=10000, help="served: requests per run")
    ap.add_argument("--loads", default="1.0,0.8,0.5", help="served: offered loads (x capacity)")
    return ap.parse_args()


# --- distributed plumbing (one process per GPU; replicas, weak scaling) -------

def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def dist_init(world):
    if world <= 1:
        return None
    import torch.distributed as dist
    backend = "nccl" if __import__("torch").cuda.is_available() else "gloo"
    dist.init_process_group(backend=backend)
    return dist


def barrier(dist):
    if dist is not None:
        dist.barrier()


def max_over_ranks(dist, value: float, device) -> float:
    if dist is None:
        return value
    import torch
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# --- clocks sampled during the timed region ---------------------------------

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines: list[str] = []
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except (FileNotFoundError, OSError):
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        if self.thread:
            self.thread.join(timeout=2)
        sm, smax, reasons, power = [], [], set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.lines:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
                power.append(float(parts[3]))
            except ValueError:
                continue
            for name, val in zip(names, parts[5:9]):
                if val.lower() == "active":
                    reasons.add(name)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": max(smax),
                "power_w_max": max(power) if power else None, "samples": len(sm),
                "reasons": sorted(reasons)}


# the default kernel, its arguments, and the planning of its launch
KERNEL_FILES = ("lookahead.cu", "nq_internal.h", "search.cu")


def kernel_sha256() -> str:
    import hashlib
    h = hashlib.sha256()
    for name in KERNEL_FILES:
        with open(os.path.join(ROOT, "paper_2511_12009_gb300", "csrc", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()


def measured_traffic(n: int, d: int, layout: str):
    """Bytes per launch from the ncu capture, when it applies to this kernel and workload."""
    t = TRAFFIC_NCU
    if (t["bytes"] is None or (n, d, layout) != (t["n"], t["d"], t["layout"])
            or kernel_sha256() != t["kernel_sha256"]):
        return None
    return t["bytes"]


# --- CPU oracle baseline --------------------------------------------------------

def cpu_model() -> str:
    """The host CPU's model name (lscpu, else /proc/cpuinfo, else the machine type)."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.split(":")[0].strip() in ("Model name", "Model"):
                v = line.split(":", 1)[1].strip()
                if v and not v.isdigit():
                    vendor = ""
                    for l2 in out.splitlines():
                        if l2.split(":")[0].strip() == "Vendor ID":
                            vendor = l2.split(":", 1)[1].strip() + " "
                    return (vendor + v).strip()
    except (OSError, subprocess.SubprocessError):
        pass
    try:
        for line in open("/proc/cpuinfo"):
            if line.lower().startswith("model name"):
                return line.split(":", 1)[1].strip()
    except OSError:
        pass
    import platform
    return platform.machine()


def oracle_rate(n: int, d: int, seconds: float, seed: int = 7) -> dict:
    """The CPU oracle (all host cores, dynamic pulling) on a seeded sample of the
    same workload's subproblems, grown until it has run about `seconds`."""
    import oracle
    oracle.build()
    cols, _ = oracle.prefixes(n, d)
    rng_order = np.random.default_rng(seed).permutation(len(cols))  # seeded, no repeats
    done_nodes, done = 0, 0
    chunk = 64
    t0 = time.perf_counter()
    while time.perf_counter() - t0 < seconds and done < len(rng_order):
        idx = rng_order[done:done + chunk]
        _, nodes = oracle.count_prefixes(n, cols[idx])
        done_nodes += int(nodes.sum())
        done += len(idx)
        chunk = min(chunk * 2, 65536)
    dt = time.perf_counter() - t0
    return {"value": done_nodes / dt, "unit": UNIT, "cores": oracle.default_threads(),
            "kind": "oracle", "seconds": dt, "cpu_model": cpu_model(),
            "sample": f"{done} seeded-random subproblems of N={n}, d={d} ({done_nodes} nodes)"}


def run_reference(args):
    world, rank, _ = dist_env()
    if world > 1 and rank != 0:
        return
    n = args.n
    d = args.d or default_depth(n)
    per_step = max(1.0, min(8.0, 120.0 / max(1, args.steps + args.warmup)))
    for _ in range(args.warmup):
        oracle_rate(n, d, per_step / 4, seed=1)
    rates, total_nodes, total_s = [], 0, 0.0
    for k in range(args.steps):
        r = oracle_rate(n, d, per_step, seed=100 + k)
        rates.append(r)
        total_nodes += r["value"] * r["seconds"]
        total_s += r["seconds"]
    value = total_nodes / total_s
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": 0,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total_s / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
            "data": "synthetic", "config": {"workload": f"N={n} full count, d={d} prefixes", "n": n,
                                            "d": d},
            "cpu_baseline": {"kind": "oracle", "cores": rates[0]["cores"], "value": value,
                             "unit": UNIT, "cpu_model": cpu_model(),
                             "sample": f"each step: seeded-random subproblems of N={n}, d={d} "
                                       f"for ~{per_step:.0f} s"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# --- our arm ---------------------------------------------------------------------

def run_batched(args, device, local):
    """One graph replay over the union of N=16..21 vs six plain launches."""
    import torch
    from paper_2511_12009_gb300 import nq
    from paper_2511_12009_gb300.batch import Batch
    ns = [16, 17, 18, 19, 20, 21]
    # the autotuner's staged search over depths, layout, block / order and
    # claim chunk for the one launch (graph replays), then the tuned batch timed
    from paper_2511_12009_gb300 import tune
    tuned = tune.tune_batch(ns, reps=1)
    ds = tuned["ds"]
    best = nq.make_config(**tuned["config"])
    nodes = 0
    for n, d in zip(ns, ds):  # node counts of the tuned depths (diagnostic build, untimed)
        nodes += nq.total_ex(n, nq.make_config(d=d), nodes=True)["nodes"]
    stream = torch.cuda.current_stream(device)
    clocks = ClockSampler(local)
    with Batch(ns, ds, best) as b:
        info = b.info()
        for _ in range(max(1, min(args.warmup, 1))):
            b.run(stream)
        clocks.start()
        graph_ms, sep_ms, totals = [], [], None
        for _ in range(args.steps):
            totals, ms = b.run(stream)
            graph_ms.append(ms)
            t2, ms2 = b.run_separate(stream)
            if t2 != totals:
                raise SystemExit("batched and separate totals differ")
            sep_ms.append(ms2)
        clk = clocks.stop()
    q = json.load(open(os.path.join(ROOT, "tests", "golden", "oeis_a000170.json")))["Q"]
    exact = totals == [q[str(n)] for n in ns]
    g = float(np.mean(graph_ms))
    line = {"metric": METRIC, "value": nodes / (g * 1e-3), "unit": UNIT, "n_gpus": 1,
            "steps": args.steps, "warmup": 1, "ms_per_step": g, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
            "config": {"workload": "batched: union of N=16..21 prefix sets, one persistent "
                                   "launch replayed from a CUDA graph",
                       "ns": ns, "ds": ds, "records": info["records"], "grid": info["grid"],
                       "block": info["block"], "nodes_per_step": nodes,
                       "tuned": {"config": tuned["config"], "candidates": len(tuned["tried"]),
                                 "best_candidate_ms": tuned["ms"]},
                       "l2": "inputs resident; no flush (compute-bound, one pass)"},
            "separate_launches_ms": float(np.mean(sep_ms)),
            "graph_vs_separate": float(np.mean(sep_ms)) / g, "totals_exact": exact,
            "totals": totals, "clocks": clk, "gpu_launches": args.steps}
    print(json.dumps(line), flush=True)


def _oracle_constrained(job):
    import oracle
    n, queens = job
    return oracle.count_constrained(n, queens)[0]


def check_served_answers(reqs: list[dict], answers: dict, seed: int = 77,
                         sample: int = 384, n16: int = 16) -> dict:
    """Exactness of the served answers against references that share nothing
    with the CUDA path: every request without queens against OEIS A000170,
    and a seeded sample of the requests with queens against the CPU oracle's
    constrained backtracker (a spawned process pool, after the timed runs):
    `sample` of those with N <= 15 and `n16` with N = 16. (The oracle fills the
    rows above a fixed queen without pruning, so one N = 18 request with one
    queen costs it about six core-minutes: larger boards are checked by the
    row-sum identity instead, served_row_sums.)"""
    import multiprocessing as mp
    import synth_inputs
    q = json.load(open(os.path.join(ROOT, "tests", "golden", "oeis_a000170.json")))["Q"]
    bad = [i for i, r in enumerate(reqs) if not r["queens"] and answers[i] != q[str(r["n"])]]
    k0 = sum(1 for r in reqs if not r["queens"])
    light = [i for i, r in enumerate(reqs) if r["queens"] and r["n"] <= 15]
    mid = [i for i, r in enumerate(reqs) if r["queens"] and r["n"] == 16]
    pick = [light[j] for j in synth_inputs.sample_indices(seed, len(light), sample)]
    pick += [mid[j] for j in synth_inputs.sample_indices(seed + 1, len(mid), n16)]
    t0 = time.perf_counter()
    with mp.get_context("spawn").Pool(os.cpu_count() or 1) as pool:
        want = pool.map(_oracle_constrained, [(reqs[i]["n"], reqs[i]["queens"]) for i in pick],
                        chunksize=1)
    bad += [i for i, w in zip(pick, want) if answers[i] != w]
    return {"unconstrained_vs_oeis": k0, "constrained_vs_oracle": len(pick),
            "oracle_s": time.perf_counter() - t0, "mismatches": len(bad), "exact": not bad}


def served_row_sums(ns=(17, 18, 19, 20), seed: int = 99) -> list[dict]:
    """The row-sum identity through the server: for a seeded row r, the N
    requests "a queen at (r, c)", c = 0..N-1, partition the solutions of the
    board, so their answers add up to Q(N) (OEIS A000170)."""
    import synth_inputs
    from paper_2511_12009_gb300.serve import Server, run_stream
    q = json.load(open(os.path.join(ROOT, "tests", "golden", "oeis_a000170.json")))["Q"]
    g = synth_inputs.SplitMix64(seed)
    out = []
    with Server(max_n=20, request_slots=64, idle_ms=200) as srv:
        for n in ns:
            row = g.below(n)
            reqs = [{"id": c, "t": 0.0, "n": n, "queens": [(row, c)]} for c in range(n)]
            res = run_stream(srv, reqs, timeout_s=1800)
            got = sum(res["answers"][c] for c in range(n))
            out.append({"n": n, "row": row, "sum": got, "q": q[str(n)], "exact": got == q[str(n)]})
        srv.poll()
    return out


def run_served(args, device, local):
    """Seeded Poisson streams at fractions of the measured capacity."""
    import synth_inputs
    from paper_2511_12009_gb300.serve import Server, run_stream
    reqs = synth_inputs.request_stream(2024, args.requests, 10, 20, 0, 4, rate_per_s=1.0)
    # capacity: every request due at once
    sat = [dict(r, t=0.0) for r in reqs]
    clocks = ClockSampler(local)
    clocks.start()
    with Server(max_n=20, request_slots=64, idle_ms=200) as srv:
        res = run_stream(srv, sat, timeout_s=7200)
    capacity = len(reqs) / res["wall_s"]
    print(f"served: saturation run {res['wall_s']:.1f} s, {capacity:.2f} requests/s",
          file=sys.stderr, flush=True)
    runs = [{"load": "saturation", "wall_s": res["wall_s"], "requests_per_s": capacity,
             "p50_ms": 1e3 * float(np.percentile(list(res["latency_s"].values()), 50)),
             "p99_ms": 1e3 * float(np.percentile(list(res["latency_s"].values()), 99))}]
    answers = res["answers"]
    for load in [float(x) for x in args.loads.split(",") if x]:
        if load >= 1.0:
            continue
        rate = load * capacity
        stream = synth_inputs.request_stream(2024, args.requests, 10, 20, 0, 4, rate_per_s=rate)
        with Server(max_n=20, request_slots=64, idle_ms=200) as srv:
            r = run_stream(srv, stream, timeout_s=7200)
        lat = list(r["latency_s"].values())
        print(f"served: load {load} run {r['wall_s']:.1f} s", file=sys.stderr, flush=True)
        if r["answers"] != answers:
            raise SystemExit("answers differ between runs")
        runs.append({"load": load, "rate_per_s": rate, "wall_s": r["wall_s"],
                     "p50_ms": 1e3 * float(np.percentile(lat, 50)),
                     "p99_ms": 1e3 * float(np.percentile(lat, 99))})
    clk = clocks.stop()
    check = check_served_answers(reqs, answers)
    check["row_sums"] = served_row_sums()
    check["exact"] = check["exact"] and all(x["exact"] for x in check["row_sums"])
    line = {"metric": METRIC, "value": capacity, "unit": "requests/s", "n_gpus": 1,
            "steps": len(runs), "warmup": 0, "ms_per_step": 1e3 * runs[0]["wall_s"],
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
            "data": "synthetic",
            "config": {"workload": f"served: {len(reqs)} seeded requests, N uniform in [10, 20], "
                                   "0-4 non-attacking queens, Poisson arrivals",
                       "request_slots": 64, "stack_slots": 13},
            "runs": runs, "answers": check, "answers_exact": check["exact"], "clocks": clk}
    print(json.dumps(line), flush=True)


def run_probe27(args, device, local):
    """4096 seeded N=27 subtrees (uniform ranks at d=8, 2-row seeded extension)."""
    import torch
    import synth_inputs
    from paper_2511_12009_gb300 import nq
    n, d0, extra, k = 27, 8, 2, 4096
    total = nq.prefix_count(n, d0)
    ranks = synth_inputs.sample_ranks(27, total, k + 256)
    choices = synth_inputs.raw_u64(2700, k + 256)
    picked = []
    for i, p in enumerate(nq.prefixes_at_ranks(n, d0, ranks)):
        kids = nq.descendants(p, extra)
        if len(kids):
            picked.append(kids[choices[i] % len(kids)])
        if len(picked) == k:
            break
    host_pre = np.array(picked, dtype=nq.PREFIX_DTYPE)
    pre = nq.to_device(host_pre, device)
    cnt = torch.zeros(k, dtype=torch.int64, device=device)
    nod = torch.zeros(k, dtype=torch.int64, device=device)
    nq.count_ex(pre, d0 + extra, n, cnt, nod, None, None)
    nq.sync()
    nodes = int(nod.cpu().numpy().view(np.uint64).sum())
    want = cnt.cpu().numpy().view(np.uint64).copy()
    stream = torch.cuda.current_stream(device)
    clocks = ClockSampler(local)
    # as device records: 4096 heavy subproblems on ~10^5 resident lanes (the default
    # form splits them by itself)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    nq.count(n, d0 + extra, pre, cnt, stream)
    nq.sync(stream)
    e0.record(stream)
    for _ in range(args.steps):
        nq.count(n, d0 + extra, pre, cnt, stream)
    e1.record(stream)
    nq.sync(stream)
    direct_ms = e0.elapsed_time(e1) / args.steps
    # the same launch with subtree donation (idle lanes take shallow frames of busy ones;
    # donation is built for the REG and REGM forms, so REGM here)
    don_cfg = nq.make_config("regm", donate=2)
    cnt_d = torch.zeros(k, dtype=torch.int64, device=device)
    nq.count_ex(pre, d0 + extra, n, cnt_d, None, None, don_cfg, stream)
    nq.sync(stream)
    donate_exact = np.array_equal(cnt_d.cpu().numpy().view(np.uint64), want)
    e0.record(stream)
    for _ in range(args.steps):
        nq.count_ex(pre, d0 + extra, n, cnt_d, None, None, don_cfg, stream)
    e1.record(stream)
    nq.sync(stream)
    donate_ms = e0.elapsed_time(e1) / args.steps
    # as host records, through nq_count_split
    split = nq.count_split(host_pre, -1)
    clocks.start()
    runs = [nq.count_split(host_pre, -1) for _ in range(args.steps)]
    clk = clocks.stop()
    exact = all(np.array_equal(r["counts"], want) for r in [split] + runs)
    ms = min(r["kernel_ms"] for r in runs)
    line = {"metric": METRIC, "value": nodes / (ms * 1e-3), "unit": UNIT, "n_gpus": 1,
            "steps": args.steps, "warmup": 1, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
            "config": {"workload": "N=27 probe: 4096 seeded depth-10 subtrees", "n": n,
                       "nodes_per_step": nodes, "solutions": int(want.sum()),
                       "split_rows": split["rows"], "split_children": split["children"],
                       "split_host_ms": min(r["split_ms"] for r in runs),
                       "split_call_ms": min(r["total_ms"] for r in runs),
                       "unsplit_kernel_ms": direct_ms, "counts_equal_unsplit": exact,
                       "donation_kernel_ms": donate_ms, "donation_counts_exact": donate_exact},
            "clocks": clk, "gpu_launches": args.steps}
    print(json.dumps(line), flush=True)


def roofline_of(nodes: int, launch_s: float, sms: int, sm_max_mhz: float) -> dict:
    """Integer roofline of one search launch: algorithmic 32-bit ops (10 per
    node) per second against the SM's integer issue capacity."""
    achieved = nodes * ALU_OPS_PER_NODE / launch_s / 1e12
    peak = sms * sm_max_mhz * 1e6 * INT_LANES_PER_CLK_SM / 1e12
    peak_alu = sms * sm_max_mhz * 1e6 * ALU_PIPE_LANES_PER_CLK_SM / 1e12
    return {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "Tops/s",
            "frac": achieved / peak, "traffic": None, "ops_per_node": ALU_OPS_PER_NODE,
            "nodes_per_launch": nodes,
            "peak_basis": f"{sms} SMs x {sm_max_mhz:.0f} MHz x {INT_LANES_PER_CLK_SM} int32 "
                          f"lanes/clk/SM (ALU pipe 64 + FMA pipe 64 = the issue rate)",
            "peak_alu_pipe": peak_alu, "frac_alu_pipe": achieved / peak_alu}


def solve_n22(args, sms: int, sm_max: float, local: int) -> dict:
    """Q(22) through nq_total_ex with the default configuration: solve time end
    to end and the search kernel's own time (CUDA events on its stream)."""
    from paper_2511_12009_gb300 import nq
    q = json.load(open(os.path.join(ROOT, "tests", "golden", "oeis_a000170.json")))["Q"]
    nodes = N22_D7_NODES
    if args.n22_nodes:
        nodes = nq.total_ex(22, nq.make_config(d=7), nodes=True)["nodes"]
    clocks = ClockSampler(local)
    clocks.start()
    t0 = time.perf_counter()
    r = nq.total_ex(22)
    wall = time.perf_counter() - t0
    clk = clocks.stop()
    if r["total"] != q["22"]:
        raise SystemExit(f"N=22 total {r['total']} != {q['22']}")
    if r["d"] != 7:
        raise SystemExit("the N=22 node count is for depth 7")
    kern_s = r["kernel_ms"] * 1e-3
    return {"total": r["total"], "exact": True, "d": r["d"], "subproblems": r["prefixes"],
            "solve_ms": 1e3 * wall, "kernel_ms": r["kernel_ms"],
            "enumerate_ms": r["enumerate_ms"], "nodes": nodes,
            "nodes_counted_now": bool(args.n22_nodes),
            "value": nodes / kern_s, "e2e_value": nodes / wall, "unit": UNIT,
            "roofline": roofline_of(nodes, kern_s, sms, sm_max), "clocks": clk,
            "paper_ms": 216740, "paper_hw": "1x RTX 4090 (Table 6, best configuration)"}


def solve_n14(reps: int = 50) -> dict:
    """The smallest configured workload, N = 14 at the library's depth: a
    latency probe. `reps` exact solves through nq_total_ex (enumerate, upload,
    search, total back), median wall and kernel times."""
    from paper_2511_12009_gb300 import nq
    nq.total_ex(14)  # warm
    walls, kerns, exact = [], [], True
    for _ in range(reps):
        t0 = time.perf_counter()
        r = nq.total_ex(14)
        walls.append(1e3 * (time.perf_counter() - t0))
        kerns.append(r["kernel_ms"])
        exact = exact and r["total"] == 365596
    return {"workload": f"N=14 full count, d={r['d']} ({r['prefixes']} subproblems)",
            "reps": reps, "solve_ms_median": float(np.median(walls)),
            "kernel_ms_median": float(np.median(kerns)), "exact": exact}


def quick_batched() -> dict:
    """The batched form beside the plain one, short: one graph replay over the
    union of N=16..21 (library depths and launch defaults) and the same work as
    six plain launches, each timed by CUDA events; totals against OEIS."""
    from paper_2511_12009_gb300.batch import Batch
    q = json.load(open(os.path.join(ROOT, "tests", "golden", "oeis_a000170.json")))["Q"]
    ns = [16, 17, 18, 19, 20, 21]
    with Batch(ns, None, None) as b:
        info = b.info()
        totals, graph_ms = b.run()
        t2, sep_ms = b.run_separate()
    return {"workload": "union of N=16..21 prefix sets, one persistent launch from a CUDA graph",
            "records": info["records"], "graph_ms": graph_ms, "separate_launches_ms": sep_ms,
            "graph_vs_separate": sep_ms / graph_ms,
            "totals_exact": totals == t2 == [q[str(n)] for n in ns]}


def quick_served(requests: int = 300) -> dict:
    """The served form, short: a seeded stream of `requests` (N uniform in
    [10, 20], 0-4 queens) all due at once; requests/s and latency; answers
    without queens against OEIS and the row-sum identity at N = 17, 18."""
    import synth_inputs
    from paper_2511_12009_gb300.serve import Server, run_stream
    q = json.load(open(os.path.join(ROOT, "tests", "golden", "oeis_a000170.json")))["Q"]
    reqs = [dict(r, t=0.0) for r in synth_inputs.request_stream(2024, requests, 10, 20, 0, 4, 1.0)]
    with Server(max_n=20, request_slots=64, idle_ms=200) as srv:
        res = run_stream(srv, reqs, timeout_s=900)
        srv.poll()
    lat = list(res["latency_s"].values())
    bad = [i for i, r in enumerate(reqs)
           if not r["queens"] and res["answers"][i] != q[str(r["n"])]]
    sums = served_row_sums(ns=(17, 18))
    return {"workload": f"{requests} seeded requests, N uniform in [10, 20], 0-4 queens, "
                        "all due at once", "requests_per_s": requests / res["wall_s"],
            "wall_s": res["wall_s"], "p50_ms": 1e3 * float(np.percentile(lat, 50)),
            "p99_ms": 1e3 * float(np.percentile(lat, 99)),
            "unconstrained_vs_oeis": sum(1 for r in reqs if not r["queens"]),
            "row_sums": sums, "exact": not bad and all(x["exact"] for x in sums)}


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    if args.workload != "n18":
        import torch
        world, rank, local = dist_env()
        torch.cuda.set_device(local)
        device = torch.device("cuda", local)
        fn = {"batched": run_batched, "served": run_served, "probe27": run_probe27}[args.workload]
        return fn(args, device, local)
    import torch
    from paper_2511_12009_gb300 import nq

    world, rank, local = dist_env()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (there is no CPU fallback)")
    torch.cuda.set_device(local)
    device = torch.device("cuda", local)
    dist = dist_init(world)
    lib = nq.lib()
    del lib
    n = args.n
    d = args.d or nq.default_depth(n)
    cfg = nq.make_config(args.layout, args.block, args.bps, args.order, d)
    stream = torch.cuda.Stream(device)

    # inputs resident in HBM
    pre_h = nq.enumerate_prefixes(n, d)
    pre = nq.to_device(pre_h, device)
    m = len(pre_h)
    counts = torch.zeros(m, dtype=torch.int64, device=device)
    totals = torch.zeros(32, dtype=torch.int64, device=device)
    flush = torch.empty(256 * 1024 * 1024, dtype=torch.uint8, device=device)

    # nodes of this workload: the diagnostic build counts them once, untimed
    nodes_t = torch.zeros(m, dtype=torch.int64, device=device)
    with torch.cuda.stream(stream):
        totals.zero_()
        nq.count_ex(pre, d, n, counts, nodes_t, totals, cfg, stream)
    nq.sync(stream)
    nodes_per_step = int(nodes_t.cpu().numpy().view(np.uint64).sum())
    total_q = int(totals.cpu().numpy().view(np.uint64)[n])
    del nodes_t

    def step():
        totals.zero_()
        nq.count_ex(pre, d, n, counts, None, totals, cfg, stream)

    with torch.cuda.stream(stream):
        for _ in range(args.warmup):
            step()
    nq.sync(stream)
    if int(totals.cpu().numpy().view(np.uint64)[n]) != total_q:
        raise SystemExit("warm-up total differs from the first run")

    clocks = ClockSampler(local)
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    barrier(dist)
    torch.cuda.synchronize(device)
    clocks.start()
    time.sleep(0.3)
    t_wall0 = time.perf_counter()
    with torch.cuda.stream(stream):
        for k in range(args.steps):
            flush.zero_()  # L2 (129 MB) flushed between steps, outside the timed events
            starts[k].record(stream)
            step()
            ends[k].record(stream)
    torch.cuda.synchronize(device)
    t_wall = time.perf_counter() - t_wall0
    barrier(dist)
    clk = clocks.stop()
    rc = nq.lib().nq_sync(stream.cuda_stream)
    if rc != 0:
        raise SystemExit(f"search reported {nq.strerror(rc)}")
    step_ms = [s.elapsed_time(e) for s, e in zip(starts, ends)]
    kern_s = sum(step_ms) * 1e-3
    kern_s_max = max_over_ranks(dist, kern_s, device)
    if int(totals.cpu().numpy().view(np.uint64)[n]) != total_q:
        raise SystemExit("timed total differs from the first run")
    value = nodes_per_step * args.steps * world / kern_s_max
    ms_per_step = 1e3 * kern_s_max / args.steps

    # end to end through the public C call (enumerate, H2D, search, D2H)
    e2e = None
    if args.e2e_steps > 0:
        e2e_times = []
        e2e_cfg = nq.make_config(args.layout, args.block, args.bps, args.order, args.d)
        for k in range(args.e2e_steps + 1):
            t0 = time.perf_counter()
            r = nq.total_ex(n, e2e_cfg)
            dt = time.perf_counter() - t0
            if r["total"] != total_q:
                raise SystemExit("end-to-end total differs")
            if k:  # the first call warms the pinned staging buffer
                e2e_times.append(dt)
        e2e_s = max_over_ranks(dist, float(np.mean(e2e_times)), device)
        # The default form copies the first four rows' prefixes (a chosen depth's whole set)
        # and a 272-byte head, which comes back; the others copy the whole set and read one
        # total.
        splits = args.layout in ("default", "regp")
        records = nq.prefix_count(n, min(d, 4)) if splits and not args.d else m
        e2e = {"value": nodes_per_step * world / e2e_s, "unit": UNIT,
               "h2d_bytes_per_step": records * 16 + (272 if splits else 0),
               "d2h_bytes_per_step": 272 if splits else 8,
               "solve_ms": 1e3 * e2e_s, "enumerate_ms": r["enumerate_ms"],
               "upload_ms": r["upload_ms"]}

    # roofline of the one kernel: algorithmic int ops per launch / launch time
    props = torch.cuda.get_device_properties(device)
    sms = props.multi_processor_count
    peaks = {}
    try:
        peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except (OSError, ValueError):
        pass
    sm_max = float(peaks.get("sm_max_mhz") or clk.get("sm_max_mhz") or SM_MAX_MHZ_FALLBACK)
    roofline = roofline_of(nodes_per_step, kern_s_max / args.steps, sms, sm_max)
    roofline["traffic"] = measured_traffic(n, d, args.layout)

    # N = 22: one exact solve through the public call, timed whole (enumeration,
    # upload, search, total back)
    n22 = None
    if rank == 0 and not args.no_n22 and args.n == 18:
        n22 = solve_n22(args, sms, sm_max, local)
    # short batched and served measurements (a failure is recorded, not fatal:
    # the line above is the benchmark)
    extras = {}
    if rank == 0 and not args.no_extras and args.n == 18:
        for name, fn in (("n14", solve_n14), ("batched", quick_batched),
                         ("served", quick_served)):
            try:
                extras[name] = fn()
            except Exception as e:  # noqa: BLE001
                extras[name] = {"error": f"{type(e).__name__}: {e}"}

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = oracle_rate(n, d, args.cpu_seconds)

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_per_step,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
                "data": "synthetic",
                "config": {"workload": f"N={n} full count, d={d} prefixes ({m} subproblems)",
                           "n": n, "d": d, "subproblems": m, "nodes_per_step": nodes_per_step,
                           "layout": args.layout, "block": args.block, "blocks_per_sm": args.bps,
                           "order": args.order,
                           "nodes": "queen placements of Algorithm 2's tree below the prefixes "
                                    "(the oracle's node count); the default form's look-ahead "
                                    "finds the same solutions in fewer steps",
                           "l2": "flushed between steps (256 MiB write outside the timed events)",
                           "parallelism": f"replicas x{world}"},
                "solve_ms": ms_per_step, "total": total_q, "wall_s": t_wall,
                "roofline": roofline, "cpu_baseline": cpu, "e2e": e2e, "clocks": clk,
                "n22": n22, **extras, "gpu_launches": args.steps}
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
