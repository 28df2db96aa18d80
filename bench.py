#!/usr/bin/env python
"""Benchmark: time to exact omega and edges/s on the R-MAT scale-22 workload.

One step = one exact maximum-clique solve through the C ABI (core numbers,
heuristic, pruning, search, witness verification, omega and witness back on
the host) of a device-resident CSR: R-MAT scale 22, edge factor 16,
(a, b, c) = (0.57, 0.19, 0.19), planted clique of 40, seed 2 (4.19M vertices,
64.2M edges; the 537 MB CSR is larger than L2, so no flush is needed).
Reported: value = undirected edges / seconds to exact omega (whole job, all
ranks), e2e = the same through host buffers with the host->device copy of the
CSR inside the timed region, roofline of the dominant kernel, the CPU oracle on
a bounded sample, clocks sampled during the timed region.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "s to exact omega & edges/s (GPU, chosen vs plain B&B); HBM GB/s frac of peak"
UNIT = "edges/s"
SAMPLE_SCALE = 15  # CPU oracle sample: same R-MAT generator at scale 15


def load_peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "fallback": True}


# Per-solve DRAM traffic (dram__bytes_read.sum + dram__bytes_write.sum) of
# the kernels on the R-MAT scale-22 solve, from one ncu capture of the
# current kernels; None until captured (and again whenever a kernel changes).
# search_block_kernel: its 512-, 864- and 1,024-candidate launches of one solve,
# 250.37 + 4.00 MB, 6.29 + 0 MB and 6.36 + 0 MB.
TRAFFIC_S22 = {"search_block_kernel": 267.02e6}


def roofline(stats, n, nnz, clk, dev):
    """Roofline of the kernel that takes the most time in a solve, timed by the
    library's CUDA events on its own stream over the timed steps.

    - kcore_peel_kernel: HBM-bound; algorithmic bytes = the CSR read once plus
      the core numbers written, 8(n+1) + 4 nnz + 4n.
    - heuristic_kernel: against HBM; algorithmic bytes = 4 B per row entry
      read and per adjacency test (mc_stats counts both).
    - search_block_kernel / search_warp_kernel (InitialBranch + Branch):
      bound by shared-memory probes, one per later-neighbour row entry read
      while building the neighbourhood matrices (Fact 3's work); peak = SMs x
      32 lanes x SM clock, one 4-byte shared-memory access per lane per clock.
    - anything else: HBM-bound against the CSR read once.
    """
    import torch
    peaks = load_peaks()
    mean = lambda k: sum(s[k] for s in stats) / len(stats)
    kern = {
        "kcore_peel_kernel": mean("ms_cores"),
        "heuristic_kernel": mean("ms_heuristic"),
        "prune (outdeg, fill, scans)": mean("ms_prune"),
        "search_block_kernel": mean("ms_search_block"),
        "search_block_kernel (big neighbourhoods)": mean("ms_search_big"),
        "search_warp_kernel": mean("ms_search_warp"),
        "branch_task_kernel": mean("ms_search_tasks"),
        "verify": mean("ms_verify"),
    }
    dom = max(kern, key=kern.get)
    ms = kern[dom]
    hbm_peak = peaks.get("hbm_gbs", 6800.0)
    hbm_src = "MEASURED_PEAKS.json hbm_gbs (of measured)" if not peaks.get("fallback") else "fallback 6.8 TB/s"
    streaming = streaming_fractions(stats, n, nnz, hbm_peak)
    if dom in ("search_block_kernel", "search_warp_kernel"):
        ent = mean("neighbourhood_entries_block") if dom == "search_block_kernel" else \
            mean("neighbourhood_entries") - mean("neighbourhood_entries_block")
        sms = torch.cuda.get_device_properties(dev).multi_processor_count
        mhz = clk.get("sm_max_mhz") or 2070.0
        peak = sms * 32 * mhz * 1e6 / 1e9
        achieved = ent / (ms / 1e3) / 1e9
        return {"bound": "alu", "kernel": dom, "achieved": achieved, "peak": peak, "unit": "G entries/s",
                "frac": achieved / peak,
                "traffic": TRAFFIC_S22.get(dom),
                "peak_source": "derived: %d SMs x 32 lanes x %.0f MHz, one shared-memory probe per lane per clock"
                               % (sms, mhz),
                "algorithmic_units": ent, "unit_note": "look-ups that build the matrices of InitialBranch (Fact 3): neighbour-list "
                "entries read, or member pairs gathered from bit rows",
                "kernel_ms": ms, "streaming": streaming, "_stages": kern}
    if dom == "heuristic_kernel":
        # Algorithm 1's reads: every row entry it scans and one 4-byte column
        # word per adjacency test (O(|E| Delta), Section 4.1)
        alg = 4 * (mean("heuristic_row_entries") + mean("heuristic_tests"))
        note = "4 B per CSR row entry read and per adjacency test of the greedy steps (mostly L2-served)"
    else:
        alg = 8 * (n + 1) + 4 * nnz + (4 * n if dom == "kcore_peel_kernel" else 0)
        note = "the CSR read once" + (" and the core numbers written" if dom == "kcore_peel_kernel" else "")
    achieved = alg / (ms / 1e3) / 1e9
    return {"bound": "hbm", "kernel": dom, "achieved": achieved, "peak": hbm_peak, "unit": "GB/s",
            "frac": achieved / hbm_peak, "traffic": TRAFFIC_S22.get(dom),
            "peak_source": hbm_src, "algorithmic_bytes": alg,
            "unit_note": note, "kernel_ms": ms, "streaming": streaming, "_stages": kern}


def streaming_fractions(stats, n, nnz, hbm_peak):
    """Achieved HBM bandwidth of the streaming phases against the measured
    copy peak, from algorithmic bytes over each stage's CUDA-event time:
    - core numbers: the CSR read once and K written, 8(n+1) + 4 nnz + 4n;
    - pruning: the keep flags scanned (8 n), the kept rows read with one
      new-id lookup per entry (8 per entry), the oriented rows written (4
      per arc);
    - heuristic: 4 B per row entry read and per adjacency test.
    """
    mean = lambda k: sum(s.get(k, 0) for s in stats) / len(stats)
    out = {}
    parts = {
        "kcore_peel_kernel": (mean("ms_cores"), 8 * (n + 1) + 4 * nnz + 4 * n),
        "prune": (mean("ms_prune"), 8 * n + 8 * mean("prune_row_entries") + 4 * mean("pruned_arcs")),
        "heuristic": (mean("ms_heuristic"), 4 * (mean("heuristic_row_entries") + mean("heuristic_tests"))),
    }
    for k, (ms, b) in parts.items():
        if ms > 0:
            gbs = b / (ms / 1e3) / 1e9
            out[k] = {"ms": ms, "algorithmic_bytes": b, "achieved_gbs": gbs, "frac": gbs / hbm_peak}
    return out



def max_over_ranks(x: float, device) -> float:
    """The largest x over all ranks of the initialised process group (x
    itself on one rank); device: where the reduction tensor lives (cuda for
    NCCL, cpu for gloo)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_value(units_per_rank: float, ranks: int, ms_max: float) -> float:
    """Whole-job throughput: the units every rank processed over the slowest
    rank's time (weak scaling: every rank solves its own replica)."""
    return units_per_rank * ranks / (ms_max / 1e3)


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons (200 ms)."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu: int, path: str | None = None):
        """path: where the raw samples go (a temporary file if None)."""
        self.gpu = gpu
        self.proc = None
        if path is None:
            import tempfile
            fd, path = tempfile.mkstemp(prefix="clocks_gpu%d_" % gpu, suffix=".csv")
            os.close(fd)
        self.path = path

    def start(self):
        try:
            if os.path.dirname(self.path):
                os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits",
                                          "-lms", "200", "-i", str(self.gpu)], stdout=self.f,
                                         stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(5)
        except Exception:
            self.proc.kill()
        self.f.close()
        mhz, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            p = [x.strip() for x in line.split(",")]
            if len(p) < 9:
                continue
            try:
                mhz.append(float(p[1]))
                mx = float(p[2])
            except ValueError:
                continue
            for nm, v in zip(names, p[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        mhz.sort()
        med = mhz[len(mhz) // 2] if mhz else None
        return {"sm_mhz": med, "sm_max_mhz": mx, "reasons": sorted(reasons), "samples": len(mhz)}


def host_info():
    """Host CPU model and logical core count (the CPU baseline's machine)."""
    model = None
    try:
        for line in open("/proc/cpuinfo"):
            if line.lower().startswith("model name"):
                model = line.split(":", 1)[1].strip()
                break
    except OSError:
        pass
    if model is None:
        try:
            out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
            for line in out.splitlines():
                if line.startswith("Model name") or line.startswith("Vendor ID"):
                    model = line.split(":", 1)[1].strip()
                    if line.startswith("Model name"):
                        break
        except Exception:
            pass
    return {"nproc": os.cpu_count(), "cpu_model": model}


def oracle_threads() -> int:
    """The host cores the CPU baseline uses: all of them (at most 64)."""
    return max(1, min(64, os.cpu_count() or 1))


def oracle_sample(seconds_min: float = 10.0, max_runs: int = 50):
    """The CPU oracle as it stands (its search with one worker per host core
    sharing the incumbent, Section 4.5) on the bounded sample (same
    generator)."""
    import oracle
    import graphgen as gg
    g = gg.rmat(SAMPLE_SCALE, 16, 0.57, 0.19, 0.19, planted=40, seed=2)
    th = oracle_threads()
    runs, tot = 0, 0.0
    while runs < max_runs and (tot < seconds_min or runs == 0):
        t = time.perf_counter()
        om, wit, st = oracle.max_clique_threads(g, th)
        tot += time.perf_counter() - t
        runs += 1
    return {"value": g.m * runs / tot, "unit": UNIT, "cores": th, "kind": "oracle", "host": host_info(),
            "sample": "oracle (%d threads) on R-MAT scale %d ef 16 (0.57,0.19,0.19) planted 40 seed 2 "
                      "(n=%d, m=%d, omega=%d), %d run(s), %.1f s" % (th, SAMPLE_SCALE, g.n, g.m, om, runs, tot)}


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return
    import oracle
    import graphgen as gg
    from graphgen import workloads as W
    g = gg.rmat(SAMPLE_SCALE, 16, 0.57, 0.19, 0.19, planted=40, seed=2)
    th = oracle_threads()
    for _ in range(args.warmup):
        oracle.max_clique_threads(g, th)
    t = time.perf_counter()
    for _ in range(args.steps):
        om, _, _ = oracle.max_clique_threads(g, th)
    dt = time.perf_counter() - t
    value = g.m * args.steps / dt
    sample = ("oracle (as it stands, %d threads sharing the incumbent) on R-MAT scale %d ef 16 (0.57,0.19,0.19) "
              "planted 40 seed 2 (n=%d, m=%d, omega=%d), one solve per step" % (th, SAMPLE_SCALE, g.n, g.m, om))
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1e3 / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "int32", "data": "synthetic",
        "config": {"workload": W.RMAT_S22,
                   "sample": "each step: the oracle on R-MAT scale %d from the same generator (n=%d, m=%d); "
                             "the scale-22 solve takes the single-thread oracle 6,161 s" % (SAMPLE_SCALE, g.n, g.m)},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": th, "kind": "oracle", "sample": sample,
                         "host": host_info()},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }), flush=True)


def _timed(solve, stream, steps, warmup):
    """Mean ms of `steps` solves after `warmup` untimed ones (CUDA events on
    the library's stream) and the last result."""
    import torch
    for _ in range(warmup):
        res = solve()
    torch.cuda.synchronize()
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    t0.record(stream)
    out = []
    for _ in range(steps):
        out.append(solve())
    t1.record(stream)
    torch.cuda.synchronize()
    return t0.elapsed_time(t1) / steps, out


def _pick_heuristic(solve_with, stream, trials=2, extents=(0, 3)):
    """The faster Algorithm 1 extent for an arm: the full algorithm (0) or
    its warm-up part only (3), each timed over `trials` solves after one
    untimed solve; omega is exact either way."""
    best = None
    for hv in extents:
        ms, _ = _timed(lambda: solve_with(hv), stream, trials, 1)
        if best is None or ms < best[1]:
            best = (hv, ms)
    return best[0]


def _load_net(args):
    import numpy as np
    import paper_1302_6256_gb300 as mc
    net = mc.MLP(seed=0)
    net.set_params(np.load(args.weights))
    return net


def run_batch(args):
    """The Erdos-Renyi batch: one plain solve per graph, the batched solve
    (one persistent pipeline for all graphs, CUDA-graph replay) and the
    learned batched solve; every omega checked against the oracle's stored
    values when available."""
    import numpy as np
    import torch
    import paper_1302_6256_gb300 as mc
    from graphgen import workloads as W

    mc.load_library()
    b = W.er_batch_4096(args.batch_count)
    dev = torch.device("cuda", 0)
    stream = torch.cuda.current_stream(dev)
    gold = os.path.join(ROOT, "tests", "golden", "er-batch-%d.json" % args.batch_count)
    ref = np.array(json.load(open(gold))["omegas"], np.int32) if os.path.exists(gold) else None
    arms = {}
    if args.form in ("per-graph", "all"):
        hs = [mc.mc_load_csr(torch.from_numpy(g.row_ptr).to(dev), torch.from_numpy(g.col_idx).to(dev), 0,
                             stream=stream) for g in b.graphs]
        # one plain solve per graph: direct launches, no task queue
        ms, res = _timed(lambda: np.array([mc.mc_max_clique(x, no_split=True)[0] for x in hs], np.int32), stream,
                         max(1, min(args.steps, 2)), 1)
        arms["per-graph"] = {"ms": ms, "omegas": res[-1], "options": "one plain solve per graph"}
        for x in hs:
            x.close()
    h = mc.mc_load_batch(torch.from_numpy(b.voff).to(dev), torch.from_numpy(b.row_ptr).to(dev),
                         torch.from_numpy(b.col_idx).to(dev), 0, stream=stream)
    net = _load_net(args) if args.form in ("learned", "all") else None
    forms = [f for f in ("chosen", "learned") if args.form in (f, "all")]
    for f in forms:
        base = dict(graph=True) if f == "chosen" else dict(graph=True, mlp=net)
        hv = _pick_heuristic(lambda x: mc.mc_max_clique_batch(h, heuristic=x, **base), stream,
                             extents=args.chosen_extents if f == "chosen" else args.learned_extents)
        opts = dict(base, heuristic=hv)
        ms, res = _timed(lambda: mc.mc_max_clique_batch(h, **opts), stream, args.steps, args.warmup)
        arms[f] = {"ms": ms, "omegas": res[-1][0], "stats": res[-1][2],
                   "options": {k: (v if k != "mlp" else "trained network") for k, v in opts.items()}}
    h.close()
    head = args.form if args.form in arms else forms[-1]
    out_arms = {}
    for k, a in arms.items():
        out_arms[k] = {"ms": a["ms"], "edges_per_s": b.m / (a["ms"] / 1e3), "options": a["options"],
                       "omegas_match_oracle": None if ref is None else bool(np.array_equal(ref, a["omegas"]))}
        if "stats" in a:
            out_arms[k]["stats"] = {x: a["stats"][x] for x in ("ms_cores", "ms_heuristic", "ms_learned", "ms_prune",
                                                               "ms_search", "learned_scored", "nodes")}
    ms = arms[head]["ms"]
    print(json.dumps({"metric": METRIC, "value": b.m / (ms / 1e3), "unit": UNIT, "n_gpus": 1, "steps": args.steps,
                      "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "dtype": "int32",
                      "data": "synthetic", "config": {"workload": W.ER_BATCH_4096 if args.batch_count == 4096 else
                                                      b.name, "form": head, "graphs": b.count, "n": b.n, "m": b.m,
                                                      "omega_max": int(np.max(arms[head]["omegas"]))},
                      "arms": out_arms}), flush=True)


def run_sweep(args):
    """The size sweep of the social-network recipe (the shape of the paper's
    scaling experiment): Chung-Lu graphs with Pareto exponent 2.1, mean
    degree 36, weight cap 10,000 and a planted clique of 80 (seed 5), n = 10^3
    ... 10^7 (10^8 is the chung-lu-100m workload); seconds to exact omega and
    edges/s of the default solve, device-resident CSR, CUDA events."""
    import torch
    import graphgen as gg
    import paper_1302_6256_gb300 as mc

    mc.load_library()
    dev = torch.device("cuda", 0)
    stream = torch.cuda.current_stream(dev)
    rows = []
    for e in range(3, 3 + args.sweep_points):
        n = 10 ** e
        g = gg.chung_lu(n, 2.1, 36.0, 10000.0, planted=80, seed=5)
        h = mc.mc_load_csr(torch.from_numpy(g.row_ptr).to(dev), torch.from_numpy(g.col_idx).to(dev), 0,
                           stream=stream)
        steps = args.steps if n < 10 ** 6 else 1
        ms, res = _timed(lambda: mc.mc_max_clique(h), stream, steps, 1 if n >= 10 ** 6 else args.warmup)
        om, _, st = res[-1]
        rows.append({"n": g.n, "m": g.m, "omega": om, "max_core": st["max_core"], "ms": ms,
                     "edges_per_s": g.m / (ms / 1e3), "nodes": st["nodes"], "tasks": st["tasks"],
                     "stages_ms": {k: st[k] for k in ("ms_cores", "ms_heuristic", "ms_prune", "ms_search")}})
        print(json.dumps(rows[-1]), file=sys.stderr, flush=True)
        h.close()
    last = rows[-1]
    print(json.dumps({"metric": METRIC, "value": last["edges_per_s"], "unit": UNIT, "n_gpus": 1, "steps": args.steps,
                      "warmup": args.warmup, "ms_per_step": last["ms"], "higher_is_better": True, "dtype": "int32",
                      "data": "synthetic",
                      "config": {"workload": "chung-lu sweep gamma=2.1 mean=36 cap=10000 planted=80 seed=5",
                                 "form": "default"},
                      "sweep": rows}), flush=True)


def run_order(args):
    """The clique-peeling vertex order (Section 6.2, taken in rounds) of R-MAT
    scale 22: edges/s of the order (device-resident CSR, CUDA events), its
    rounds and cliques, and the gap-coding cost (mean log2(1 + gap) bits per
    adjacency entry) of the vertex ids as generated, of the degeneracy order
    and of the clique order."""
    import numpy as np
    import torch
    import paper_1302_6256_gb300 as mc
    from graphgen import workloads as W

    mc.load_library()
    dev = torch.device("cuda", 0)
    stream = torch.cuda.current_stream(dev)
    g = W.rmat_s22()
    h = mc.mc_load_csr(torch.from_numpy(g.row_ptr).to(dev), torch.from_numpy(g.col_idx).to(dev), 0, stream=stream)
    ms, res = _timed(lambda: mc.mc_clique_order(h), stream, args.steps, args.warmup)
    order, starts, rounds, st = res[-1]
    sizes = np.diff(starts)
    peel = mc.mc_peel_order(h).copy()
    t0 = time.time()
    bits = {"ids": mc.mc_gap_bits(h), "degeneracy": mc.mc_gap_bits(h, peel), "clique": mc.mc_gap_bits(h, order)}
    gap_s = (time.time() - t0) / 3
    h.close()
    print(json.dumps({"metric": "edges/s of the clique-peeling order", "value": g.m / (ms / 1e3), "unit": "edges/s",
                      "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
                      "higher_is_better": True, "dtype": "int32", "data": "synthetic",
                      "config": {"workload": W.RMAT_S22, "n": g.n, "m": g.m, "l2": "inputs > L2 (537 MB CSR)"},
                      "rounds": st["rounds"], "cliques": int(sizes.size), "largest": int(sizes.max()),
                      "cliques_by_size": {str(k): int(v) for k, v in zip(*np.unique(np.minimum(sizes, 8),
                                                                                   return_counts=True))},
                      "grows": st["grows"], "tests": st["tests"], "ms_device": st["ms"],
                      "gap_bits": bits, "gap_call_s": gap_s}), flush=True)


def run_single(args):
    """One graph: the plain GPU B&B, the chosen form (the faster Algorithm 1
    extent) and the learned form (scores of the vertices that can beat the
    warm-up bound, seeds grown first): seconds to exact omega, the
    heuristic's lower-bound gap and the fraction of vertices pruned."""
    import numpy as np
    import torch
    import paper_1302_6256_gb300 as mc
    from graphgen import workloads as W

    mc.load_library()
    gen = {"rmat-s22": (W.RMAT_S22, W.rmat_s22), "rmat-s24": (W.RMAT_S24, W.rmat_s24),
           "chung-lu-20k": (W.CHUNG_LU_20K, W.chung_lu_20k),
           "chung-lu-100m": (W.CHUNG_LU_100M, W.chung_lu_100m)}[args.workload]
    g = gen[1]()
    dev = torch.device("cuda", 0)
    stream = torch.cuda.current_stream(dev)
    h = mc.mc_load_csr(torch.from_numpy(g.row_ptr).to(dev), torch.from_numpy(g.col_idx).to(dev), 0, stream=stream)
    wit = torch.zeros(g.n + 1, dtype=torch.int32, device=dev)
    net = _load_net(args) if args.form in ("learned", "all") else None
    forms = [f for f in ("plain", "chosen", "learned") if args.form in (f, "all")]
    arms = {}
    for f in forms:
        if f == "plain":
            opts = dict(no_split=True)
        else:
            base = {} if f == "chosen" else dict(mlp=net)
            hv = _pick_heuristic(lambda x: mc.mc_max_clique(h, witness_out=wit, heuristic=x, **base), stream,
                                 extents=args.chosen_extents if f == "chosen" else args.learned_extents)
            opts = dict(base, heuristic=hv)
        ms, res = _timed(lambda: mc.mc_max_clique(h, witness_out=wit, **opts), stream, args.steps, args.warmup)
        om, _, st = res[-1]
        hs = sum(r[2]["heuristic_size"] for r in res) / len(res)
        arms[f] = {"ms": ms, "edges_per_s": g.m / (ms / 1e3), "omega": om,
                   "options": {k: (v if k != "mlp" else "trained network") for k, v in opts.items()},
                   "heuristic_mean": hs, "lower_bound_gap": om - hs, "fraction_pruned": 1.0 - st["pruned_n"] / g.n,
                   "stats": {k: st[k] for k in ("ms_total", "ms_cores", "ms_heuristic", "ms_learned", "ms_prune",
                                                "ms_search", "learned_scored", "pruned_n", "nodes",
                                                "neighbourhood_entries", "max_core")}}
    assert len({a["omega"] for a in arms.values()}) == 1
    head = args.form if args.form in arms else forms[-1]
    ms = arms[head]["ms"]
    print(json.dumps({"metric": METRIC, "value": g.m / (ms / 1e3), "unit": UNIT, "n_gpus": 1, "steps": args.steps,
                      "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "dtype": "int32",
                      "data": "synthetic",
                      "config": {"workload": gen[0], "form": head, "n": g.n, "m": g.m, "omega": arms[head]["omega"]},
                      "arms": arms}), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--workload", default="rmat-s22",
                    choices=["rmat-s22", "er-batch", "rmat-s24", "chung-lu-20k", "chung-lu-100m", "chung-lu-sweep",
                             "clique-order"])
    ap.add_argument("--sweep-points", type=int, default=5, help="chung-lu-sweep: n = 10^3 .. 10^(2 + points)")
    ap.add_argument("--form", default="chosen", choices=["chosen", "plain", "per-graph", "learned", "all"],
                    help="chosen: the autotuned solve (on R-MAT scale 22 both arms are timed and this one is the "
                         "headline; graph replay for batches); plain: direct launches, degeneracy order, no task "
                         "queue; learned: the learned form (scores of the vertices that can beat the warm-up "
                         "bound seed the heuristic); per-graph: one solve per graph of a batch; all: every form of "
                         "the workload, the last one as the headline")
    ap.add_argument("--weights", default=os.path.join(ROOT, "paper_1302_6256_gb300", "ordering_mlp.npy"))
    ap.add_argument("--batch-count", type=int, default=4096)
    ap.add_argument("--heuristic", type=int, default=0, choices=[0, 1, 3],
                    help="override the chosen form's Algorithm 1 extent: 1 deterministic, 3 warm-up only "
                         "(0: the autotuner's choice)")
    ap.add_argument("--chosen-extents", default="0,3",
                    help="Algorithm 1 extents the chosen arm of the other workloads tries (0 full, 3 warm-up only)")
    ap.add_argument("--learned-extents", default="0,3", help="... and the learned arm")
    ap.add_argument("--clocks-csv", default=None,
                    help="keep the raw nvidia-smi samples of the timed region in this file (rank r appends _r)")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)
    args.chosen_extents = tuple(int(x) for x in args.chosen_extents.split(","))
    args.learned_extents = tuple(int(x) for x in args.learned_extents.split(","))
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "er-batch":
        return run_batch(args)
    if args.workload == "chung-lu-sweep":
        return run_sweep(args)
    if args.workload == "clique-order":
        return run_order(args)
    if args.workload != "rmat-s22" or args.form in ("learned", "all"):
        return run_single(args)

    import numpy as np
    import torch
    import torch.distributed as dist
    import paper_1302_6256_gb300 as mc
    from paper_1302_6256_gb300 import autotune
    from graphgen import workloads as W

    ws, rank, local = dist_env()
    if ws > 1:
        dist.init_process_group("nccl", init_method="env://")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    mc.load_library()

    g = W.rmat_s22()
    rp_h = torch.from_numpy(g.row_ptr).pin_memory()
    ci_h = torch.from_numpy(g.col_idx).pin_memory()
    rp = rp_h.to(dev)
    ci = ci_h.to(dev)
    torch.cuda.synchronize()
    h = mc.mc_load_csr(rp, ci, 0, stream=stream)
    wit_h = torch.zeros(g.n + 1, dtype=torch.int32).pin_memory()

    # the two forms of the metric: the plain GPU B&B (degeneracy order, no
    # task queue, direct launches, the full Algorithm 1, no learned scores)
    # and the chosen form (the autotuner's fastest setting for this workload)
    plain = dict(no_split=True)
    chosen, tune_ms, cached = autotune.tuned(h, W.RMAT_S22)
    if args.heuristic:
        chosen = dict(chosen, heuristic=args.heuristic)
    arms = {"plain": plain, "chosen": chosen}
    head = args.form if args.form in arms else "chosen"

    clocks = Clocks(local, None if args.clocks_csv is None else
                    (args.clocks_csv if ws == 1 else "%s_%d" % (args.clocks_csv, rank)))
    clocks.start()
    timed = {}
    for name in (("plain", "chosen") if head == "chosen" else ("chosen", "plain")):
        opts = arms[name]
        for _ in range(args.warmup):
            om, _, st = mc.mc_max_clique(h, witness_out=wit_h, **opts)
        if ws > 1:
            dist.barrier()
        torch.cuda.synchronize()
        launches0 = mc.mc_launch_count()
        t0 = torch.cuda.Event(enable_timing=True)
        t1 = torch.cuda.Event(enable_timing=True)
        t0.record(stream)
        stats = []
        for _ in range(args.steps):
            om, wit, st = mc.mc_max_clique(h, witness_out=wit_h, **opts)
            stats.append(st)
        t1.record(stream)
        torch.cuda.synchronize()
        if ws > 1:
            dist.barrier()
        timed[name] = {"ms": max_over_ranks(t0.elapsed_time(t1) / args.steps, dev), "stats": stats, "omega": om,
                       "launches": mc.mc_launch_count() - launches0}
    clk = clocks.stop()
    ms = timed[head]["ms"]
    stats = timed[head]["stats"]
    om = timed[head]["omega"]
    assert timed["plain"]["omega"] == timed["chosen"]["omega"]
    value = job_value(g.m, ws, ms)

    # end to end through the public API from host buffers: H2D of the CSR,
    # solve, D2H of omega and witness, every step.  Each step loads a new
    # handle and solves it once, so CUDA-graph replay (which captures on a
    # handle's first solve and pays off only on later ones) is left out here
    e2e_opts = {k: v for k, v in arms[head].items() if k != "graph"}
    e2e_steps = max(3, args.steps // 2)
    for _ in range(args.warmup):  # untimed, like the device arms' warm-up
        he = mc.mc_load_csr(rp_h, ci_h, 0, stream=stream)
        mc.mc_max_clique(he, witness_out=wit_h, **e2e_opts)
        he.close()
    torch.cuda.synchronize()
    te = time.perf_counter()
    for _ in range(e2e_steps):
        he = mc.mc_load_csr(rp_h, ci_h, 0, stream=stream)
        om_e, wit_e, _ = mc.mc_max_clique(he, witness_out=wit_h, **e2e_opts)
        he.close()
    torch.cuda.synchronize()
    e2e_ms = (time.perf_counter() - te) * 1e3 / e2e_steps
    e2e_ms = max_over_ranks(e2e_ms, dev)
    assert om_e == om

    n = g.n
    roof = roofline(stats, n, int(g.row_ptr[-1]), clk, dev)
    stages = roof.pop("_stages")
    ms_plain, ms_chosen = timed["plain"]["ms"], timed["chosen"]["ms"]

    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
        "data": "synthetic",
        "config": {"workload": W.RMAT_S22, "n": n, "m": g.m, "omega": om, "max_core": stats[-1]["max_core"],
                   "form": head,
                   "chosen_options": chosen, "chosen_from_cache": cached,
                   "plain_options": "degeneracy order, no task queue, direct launches, full Algorithm 1",
                   "ms_chosen": ms_chosen, "ms_plain": ms_plain,
                   "edges_per_s_chosen": job_value(g.m, ws, ms_chosen),
                   "edges_per_s_plain": job_value(g.m, ws, ms_plain),
                   "chosen_over_plain": ms_plain / ms_chosen,
                   "l2": "inputs > L2 (537 MB CSR)",
                   "parallelism": "replicas" if ws > 1 else "1 GPU"},
        "e2e": {"value": job_value(g.m, ws, e2e_ms), "unit": UNIT, "ms_per_step": e2e_ms,
                "h2d_bytes_per_step": int(rp_h.numel() * 8 + ci_h.numel() * 4),
                "d2h_bytes_per_step": int(4 + 4 * om),
                "options": "the chosen options without graph replay: a new handle per step, solved once"},
        "roofline": roof,
        "gpu_launches": int(timed[head]["launches"]),
        "clocks": clk,
        "kernel_ms": stages,
        "kernel_ms_plain": roofline(timed["plain"]["stats"], n, int(g.row_ptr[-1]), clk, dev)["_stages"],
        "stats_last": stats[-1],
    }
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        out["cpu_baseline"] = oracle_sample()
    if rank == 0:
        print(json.dumps(out), flush=True)
    h.close()
    if ws > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
