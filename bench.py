#!/usr/bin/env python3
"""Benchmark of the exponential-shift low-diameter decomposition on GB300.

Workload (default, --workload rmat22): R-MAT scale 22 (edge factor 16,
a,b,c,d = .57,.19,.19,.05, graph seed 7, symmetrised, self-loops and repeated
arcs removed), shifts delta_u = -ln(U_u)/beta from Philox4x32-10 seed 1, one
decomposition per beta in {0.02, 0.1, 0.5}.  One step = those three
decompositions plus the cut-edge count of each (every row of the hot path:
split, fraction rank, start buckets, BFS rounds, assignment, cut count).

Metric: GTEPS = undirected edges m x decompositions / second (Graph500
convention), whole job over all ranks.  `value` is device time with the graph
and the shifts resident in HBM (CUDA events around every step on the
library's stream; L2 flushed between steps, outside the events).  `e2e`
repeats the step through the same C ABI with host buffers (pinned), so the
shift upload, the result download and all host work are inside the clock.

The default run also measures every other configuration and nests its value under
"workloads"; the complete lines (each with its own parity check, roofline, CPU
baseline and clocks) go to stderr, one per row, so that the printed line stays
short: the 256x256 and 256^3 grids, the batch of 1,024 random geometric
graphs and the 64 seeds of one R-MAT 20 graph (decompositions/s against one
at a time), the block decomposition by repeated decomposition, and the
Poisson request stream against the server (p50/p99 against one at a time, at
the workload's rate and at rates the one-at-a-time server sustains).
--single keeps to the named workload's line (profiling commands use it).

Under torchrun (N > 1) every rank decomposes its own replica (the method has
no exchange step): value = N x per-rank work / the slowest rank's time.

--impl reference runs the CPU oracle (the method's plain definition, single
threaded) on the same workload and the same step: the three decompositions
and their cut counts.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

L2_FLUSH_BYTES = 256 << 20
FALLBACK_HBM_GBS = 6800.0


# ----------------------------------------------------------------- distributed helpers
def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def init_dist(world, backend):
    import torch.distributed as dist

    if world > 1 and not dist.is_initialized():
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        dist.init_process_group(backend)
    return dist if world > 1 else None


def barrier(dist):
    if dist is not None:
        dist.barrier()


def reduce_max(dist, x: float, device=None) -> float:
    """Max of a float over ranks (the slowest rank sets the job time)."""
    if dist is None:
        return x
    import torch

    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def reduce_sum(dist, x: float, device=None) -> float:
    if dist is None:
        return x
    import torch

    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


# ----------------------------------------------------------------- clocks
class ClockSampler:
    """nvidia-smi samples every 200 ms while the timed region runs."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except (OSError, ValueError):
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.thread.join(timeout=2)

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[4:8]):
                if val.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# ----------------------------------------------------------------- workload
def make_workload(name):
    import ldd_gen as gen

    spec = gen.WORKLOADS[name]
    t0 = time.perf_counter()
    G = gen.make_graph(spec["graph"])
    t_graph = time.perf_counter() - t0
    t0 = time.perf_counter()
    shifts = [gen.shifts(G.n, b, spec["shift_seed"]) for b in spec["betas"]]
    t_shift = time.perf_counter() - t0
    return spec, G, shifts, t_graph, t_shift


def describe(name, spec, G):
    g = spec["graph"]
    if g[0] == "rmat":
        gdesc = f"R-MAT scale {g[1]}, edge factor {g[2]}, (a,b,c)=({g[3]},{g[4]},{g[5]}), seed {g[6]}, symmetrised, dedup"
    elif g[0] == "grid3d":
        gdesc = f"3D 6-neighbour grid {g[1]}x{g[2]}x{g[3]}"
    else:
        gdesc = f"2D 4-neighbour grid {g[1]}x{g[2]}"
    return {"workload": name, "graph": gdesc, "n": G.n, "m": G.m, "nnz": G.nnz,
            "betas": list(spec["betas"]), "shift_seed": spec["shift_seed"],
            "shifts": "FP64, delta=-ln(U)/beta, U from Philox4x32-10",
            "l2": f"flushed between steps ({L2_FLUSH_BYTES >> 20} MiB write, outside the timed events)"}


def bfs_algorithmic_bytes(st):
    """Bytes the BFS kernel's executed rounds must move for one launch:
    per arc expanded top-down or scanned bottom-up 4 B of col + 8 B of the other
    end's key (probe / atomicMin); per vertex examined bottom-up 8 B of its key
    + 8 B row_ptr; per settled vertex 8 B row_ptr + 8 B own key + 24 B queue
    write and read; per start-bucket entry (one per vertex the BFS handles)
    4 B vertex id + 8 B key test.  Windows of levels may expand a vertex (and
    offer its arcs) more than once; only the first time counts here."""
    push, items = st["push_arcs"], st["items"]
    if st.get("bfs_windows", 0) > 0:
        push = min(push, st["nnz"])  # every arc offered at most once
        items = min(items, st["n_active"])
    return (12 * (push + st["pull_arcs"]) + 16 * st["pull_vertices"]
            + 40 * items + 12 * st["n_active"])


def kernel_source_sha():
    """Hash of the BFS kernel's sources (its file and the shared header)."""
    h = hashlib.sha256()
    src = os.path.join(ROOT, "paper_1307_3692_gb300", "csrc")
    for f in ("k_bfs.cu", "ldd_internal.cuh"):
        h.update(open(os.path.join(src, f), "rb").read())
    return h.hexdigest()[:16]


def ncu_traffic(workload):
    """DRAM bytes per BFS launch from the committed ncu summary, if it was taken
    on the kernels as they are now (same source hash); else None."""
    path = os.path.join(ROOT, "profiles", f"k_bfs_{workload}.md")
    if not os.path.exists(path):
        return None, None
    vals = {}
    for line in open(path):
        if ":" in line and line.strip().startswith("- "):
            k, _, v = line.strip()[2:].partition(":")
            vals[k.strip()] = v.strip().strip("`")
    sha = vals.get("source_sha")
    try:
        traffic = float(vals.get("dram_bytes_per_launch", "nan"))
    except ValueError:
        return None, sha
    if sha != kernel_source_sha() or not math.isfinite(traffic):
        return None, sha
    return traffic, sha


def measured_peak_hbm():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            v = float(json.load(f)["hbm_gbs"])
        return v, "measured"
    except (OSError, KeyError, ValueError):
        return FALLBACK_HBM_GBS, "fallback"


def gen_sample(name):
    """The workload's graph family at 1/8 of its vertices: a bounded sample
    for timing the oracle where the full size would take too long."""
    import ldd_gen as gen

    g = gen.WORKLOADS[name]["graph"]
    if g[0] == "grid3d":
        return gen.grid3d(g[1] // 2, g[2] // 2, g[3] // 2)
    if g[0] == "grid2d":
        return gen.grid2d(g[1] // 4, g[2] // 2)
    if g[0] == "rmat":
        return gen.rmat(g[1] - 3, *g[2:])
    raise ValueError(name)


def gen_shifts(n, beta, seed):
    import ldd_gen as gen

    return gen.shifts(n, beta, seed)


def step_text(betas):
    """What one step of a single-graph workload does (both arms)."""
    return f"{len(betas)} decompositions (one per beta) + their cut counts"


# ----------------------------------------------------------------- oracle (CPU) leg
def run_oracle(G, shifts_list):
    import oracle

    t0 = time.perf_counter()
    for sh in shifts_list:
        c, _ = oracle.oracle_ldd(G.row_ptr, G.col, sh)
        oracle.oracle_cut_edges(G.row_ptr, G.col, c)
    return time.perf_counter() - t0


def reference_arm(args):
    """The oracle as the reference implementation: rank 0 only."""
    world, rank, _ = dist_env()
    if rank != 0:
        return 0
    spec, G, shifts, _, _ = make_workload(args.workload)
    betas = spec["betas"]
    for i in range(args.warmup):
        run_oracle(G, shifts)
    times = []
    for i in range(args.steps):
        times.append(run_oracle(G, shifts))
    total = sum(times)
    value = len(betas) * G.m * args.steps / total / 1e9
    line = {
        "impl": "reference", "metric": "LDD GTEPS", "value": value, "unit": "GTEPS",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * total / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "u64", "data": "synthetic",
        "config": describe(args.workload, spec, G) | {"step": step_text(betas),
                                                      "parallelism": f"replicas x{world}"},
        "cpu_baseline": {"value": value, "unit": "GTEPS", "cores": 1, "host_cores": os.cpu_count(),
                         "kind": "oracle",
                         "sample": f"{args.steps} full steps ({len(betas)} decompositions + cut "
                                   f"counts each) of the {args.workload} workload, single-threaded"},
        "e2e": {"value": value, "unit": "GTEPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# ----------------------------------------------------------------- our arm
def create_info(g, wall_s):
    """Once-per-graph cost that a decomposition step amortises (ldd_create_graph)."""
    st = g.stats()
    return {"wall_ms": 1e3 * wall_s, "upload_ms": st["ms_create_upload"],
            "components_ms": st["ms_create_components"],
            "note": "once per graph, outside the timed step: CSR upload, component labelling "
                    "(device), cut-list build (host)"}


def our_arm(args, dist):
    import numpy as np
    import torch

    import paper_1307_3692_gb300 as ldd

    world, rank, local = dist_env()
    dev = torch.device("cuda", local)

    spec, G, shifts, t_graph, t_shift = make_workload(args.workload)
    betas = spec["betas"]
    n, m = G.n, G.m
    d_rp, d_col = torch.from_numpy(G.row_ptr).to(dev), torch.from_numpy(G.col).to(dev)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    g = ldd.LddGraph(d_rp, d_col, validate=False)
    create = create_info(g, time.perf_counter() - t0)
    del d_rp, d_col
    stream = torch.cuda.Stream(device=dev)
    g.set_stream(stream)
    g.set_timing(True)
    d_shifts = [torch.from_numpy(s).to(dev) for s in shifts]
    centers = [torch.empty(n, dtype=torch.int32, device=dev) for _ in betas]
    dists = [torch.empty(n, dtype=torch.int32, device=dev) for _ in betas]
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.int32, device=dev)
    torch.cuda.synchronize()

    def step():
        """One timed step: the len(betas) decompositions and their cut counts in
        one pipelined ldd_decompose_batch call on device buffers."""
        cut = g.decompose_batch(betas, d_shifts, centers, dists)
        return cut, g.stats()["launches"]

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()

    # ---- device-resident timed region
    launches = 0
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    barrier(dist)
    torch.cuda.synchronize()
    with ClockSampler(local) as clocks:
        t_wall = time.perf_counter()
        for i in range(args.steps):
            with torch.cuda.stream(stream):
                flush.fill_(i)
            ev[i][0].record(stream)
            step_cuts, l = step()
            launches += l
            ev[i][1].record(stream)
        torch.cuda.synchronize()
        t_wall = time.perf_counter() - t_wall
    barrier(dist)
    step_ms = [a.elapsed_time(b) for a, b in ev]
    local_ms = sum(step_ms) / args.steps
    ms_per_step = reduce_max(dist, local_ms, dev)
    work = len(betas) * m  # edges per step per rank
    value = world * work / (ms_per_step * 1e-3) / 1e9
    cuts = dict(zip(betas, step_cuts))

    # ---- phase breakdown (outside the timed region): the same decompositions
    # as single ldd_decompose + ldd_cut_edges calls with the library's events
    per_beta = []
    scratch_c = torch.empty(n, dtype=torch.int32, device=dev)
    scratch_d = torch.empty(n, dtype=torch.int32, device=dev)
    for _ in range(3):
        per_beta = []
        for b, sh in zip(betas, d_shifts):
            with torch.cuda.stream(stream):
                flush.fill_(0)
            g.decompose(b, sh, scratch_c, scratch_d)
            assert g.cut_edges(scratch_c) == cuts[b], "single-call cut differs from the batch"
            per_beta.append(g.stats())
    center = centers[-1]

    # ---- roofline of the dominant kernel (the persistent BFS)
    bfs_ms = [st["ms_bfs"] for st in per_beta]
    bfs_bytes = [bfs_algorithmic_bytes(st) for st in per_beta]
    avg_ms = sum(bfs_ms) / len(bfs_ms)
    avg_bytes = sum(bfs_bytes) / len(bfs_bytes)
    peak, peak_kind = measured_peak_hbm()
    achieved = avg_bytes / (avg_ms * 1e-3) / 1e9
    traffic, traffic_sha = ncu_traffic(args.workload)
    roofline = {"bound": "hbm", "kernel": "k_bfs", "achieved": achieved, "peak": peak,
                "unit": "GB/s", "frac": achieved / peak, "traffic": traffic,
                "peak_kind": f"of {peak_kind}",
                "algorithmic_bytes_per_launch": avg_bytes, "avg_launch_ms": avg_ms}
    # share of the step spent in each phase (device events inside the library)
    tot = sum(st["ms_total"] for st in per_beta) + sum(st["ms_cut"] for st in per_beta)
    phases = {k: sum(st[k] for st in per_beta) / max(tot, 1e-9) for k in
              ("ms_rank", "ms_bfs", "ms_finalize", "ms_cut")}

    # ---- end to end through the C ABI with host buffers: one pipelined batch
    # call per step (shift uploads and result downloads overlap the device work)
    h_shifts = [torch.from_numpy(s).pin_memory() for s in shifts]
    h_center = [torch.empty(n, dtype=torch.int32).pin_memory() for _ in betas]
    h_dist = [torch.empty(n, dtype=torch.int32).pin_memory() for _ in betas]
    g_e2e = ldd.LddGraph(G.row_ptr, G.col, validate=False)
    for _ in range(2):  # warm-up (also allocates the pipeline's staging)
        g_e2e.decompose_batch(betas, h_shifts, h_center, h_dist)
    barrier(dist)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        e2e_cuts = g_e2e.decompose_batch(betas, h_shifts, h_center, h_dist)
    e2e_s = (time.perf_counter() - t0) / args.steps
    barrier(dist)
    e2e_s = reduce_max(dist, e2e_s, dev)
    g_e2e.close()
    h2d = len(betas) * 8 * n                 # shifts in
    d2h = len(betas) * (8 * n + 8 + 40)      # center + dist out, cut count, status header
    e2e = {"value": world * work / e2e_s / 1e9, "unit": "GTEPS", "h2d_bytes_per_step": h2d,
           "d2h_bytes_per_step": d2h, "ms_per_step": 1e3 * e2e_s,
           "api": "ldd_decompose_batch (pinned host buffers)",
           "cuts_match_device_path": e2e_cuts == [cuts[b] for b in betas]}

    # ---- parity of the timed outputs (every beta) and CPU baseline
    cpu = None
    parity = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        import oracle

        parity = {"decompositions": len(betas), "mismatched_vertices": 0}
        big = m > 40_000_000  # the oracle's Dijkstra takes ~40 s there: certify instead
        for b, sh, c_t, d_t in zip(betas, shifts, centers, dists):
            gc, gd = c_t.cpu().numpy(), d_t.cpu().numpy()
            if big:
                code, bad = oracle.oracle_certify(G.row_ptr, G.col, sh, gc, gd)
                assert code == 0, f"timed output fails the certificate ({code}) at {bad}"
                parity["method"] = ("O(m) optimality certificate of every vertex (Lemma 3.1 "
                                    "predecessor + non-improvability) on the timed outputs")
            else:
                oc, od = oracle.oracle_ldd(G.row_ptr, G.col, sh)
                bad = int((gc != oc).sum() + (gd != od).sum())
                parity["mismatched_vertices"] += bad
                assert bad == 0, "timed output differs from the oracle"
                parity["method"] = "oracle labels, element by element, every beta of the timed step"
            assert cuts[b] == oracle.oracle_cut_edges(G.row_ptr, G.col, gc), "cut count differs"
        if big:  # the oracle timed on a bounded sample: the same family at 1/8 the size
            sample_name, S = args.workload, gen_sample(args.workload)
            t0 = time.perf_counter()
            for sh in [gen_shifts(S.n, b, spec["shift_seed"]) for b in betas]:
                oc, _ = oracle.oracle_ldd(S.row_ptr, S.col, sh)
                oracle.oracle_cut_edges(S.row_ptr, S.col, oc)
            t_cpu = time.perf_counter() - t0
            cpu = {"value": len(betas) * S.m / t_cpu / 1e9, "unit": "GTEPS", "cores": 1,
                   "host_cores": os.cpu_count(), "kind": "oracle", "seconds": t_cpu,
                   "sample": f"{len(betas)} decompositions + cut counts of {S.name} "
                             f"({S.n} vertices, {S.m} edges: the same workload at 1/8 size; "
                             "edges per second of the full size would be no higher)"}
        else:
            t_cpu = run_oracle(G, shifts)
            cpu = {"value": len(betas) * m / t_cpu / 1e9, "unit": "GTEPS", "cores": 1,
                   "host_cores": os.cpu_count(), "kind": "oracle",
                   "sample": f"one full step: {len(betas)} decompositions + cut counts of "
                             f"{args.workload}", "seconds": t_cpu}

    g.close()
    if rank == 0:
        clk = clocks.summary()
        line = {
            "metric": "LDD GTEPS", "value": value, "unit": "GTEPS", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_per_step,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "u64", "data": "synthetic",
            "config": describe(args.workload, spec, G) | {"step": step_text(betas),
                                                          "parallelism": f"replicas x{world}"},
            "api": "one pipelined ldd_decompose_batch call per step on device buffers",
            "roofline": roofline,
            "cpu_baseline": cpu,
            "e2e": e2e,
            "gpu_launches": launches,
            "clocks": {"sm_mhz": clk["sm_mhz"], "sm_max_mhz": clk["sm_max_mhz"], "reasons": clk["reasons"]},
            "per_beta": [{"beta": b, "ms_total": st["ms_total"], "ms_rank": st["ms_rank"],
                          "ms_bfs": st["ms_bfs"], "ms_finalize": st["ms_finalize"], "ms_cut": st["ms_cut"],
                          "rounds": st["rounds"], "pull_rounds": st["pull_rounds"],
                          "A": st["max_floor_shift"], "items": st["items"],
                          "push_arcs": st["push_arcs"], "pull_arcs": st["pull_arcs"],
                          "pull_vertices": st["pull_vertices"], "exact_rank": st["exact_rank"],
                          "gteps": m / st["ms_total"] / 1e6}
                         for b, st in zip(betas, per_beta[-len(betas):])],
            "phase_share": phases,
            "per_beta_source": "single ldd_decompose + ldd_cut_edges calls outside the timed region",
            "wall_s_timed_region": t_wall,
            "host_s": {"graph_generation": t_graph, "shift_draw": t_shift},
            "create_graph": create,
            "parity": parity,
            "kernel_source_sha": kernel_source_sha(),
        }
        return line
    return None


# ----------------------------------------------------------------- batched workloads
def make_batch(name):
    """(members, betas, shifts, description) of a batched workload."""
    import ldd_gen as gen

    spec = gen.BATCH_WORKLOADS[name]
    if spec["kind"] == "rgg":
        batch = gen.rgg_batch(spec["count"], spec["n_lo"], spec["n_hi"], spec["beta_lo"],
                              spec["beta_hi"], spec["master_seed"])
        Gs = [b[0] for b in batch]
        desc = (f"{spec['count']} random geometric graphs in the unit square, n uniform on "
                f"[{spec['n_lo']}, {spec['n_hi']}], mean degree 8, beta uniform on "
                f"[{spec['beta_lo']}, {spec['beta_hi']}), graph and shift seed {spec['master_seed']} + i")
        return Gs, [b[1] for b in batch], [b[2] for b in batch], desc
    G = gen.make_graph(spec["graph"])
    k = spec["copies"]
    shifts = [gen.shifts(G.n, spec["beta"], spec["first_seed"] + i) for i in range(k)]
    g = spec["graph"]
    desc = (f"{k} shift vectors (seeds {spec['first_seed']}..{spec['first_seed'] + k - 1}) of one "
            f"R-MAT scale {g[1]} graph (edge factor {g[2]}, seed {g[6]}) at beta {spec['beta']}")
    return [G] * k, [spec["beta"]] * k, shifts, desc


def batch_arm(args, dist):
    """One union decomposition of the whole batch per step, against the same
    members decomposed one at a time by ldd_decompose on the same GPU."""
    import numpy as np
    import torch

    import paper_1307_3692_gb300 as ldd

    world, rank, local = dist_env()
    dev = torch.device("cuda", local)
    t0 = time.perf_counter()
    Gs, betas, shifts, desc = make_batch(args.workload)
    t_gen = time.perf_counter() - t0
    k = len(Gs)
    t0 = time.perf_counter()
    uniq = {}
    for G in Gs:  # one member graph object per distinct graph
        if id(G) not in uniq:
            uniq[id(G)] = ldd.LddGraph(torch.from_numpy(G.row_ptr).to(dev),
                                       torch.from_numpy(G.col).to(dev), validate=False)
    members = [uniq[id(G)] for G in Gs]
    u = ldd.LddUnion(members)
    t_create = time.perf_counter() - t0
    stream = torch.cuda.Stream(device=dev)
    u.set_stream(stream)
    u.set_timing(True)
    u.set_graph_replay(not args.no_replay)
    for m in uniq.values():
        m.set_stream(stream)
    total = u.total
    m_total = sum(G.m for G in Gs)
    d_shift = torch.from_numpy(np.concatenate(shifts)).to(dev)
    center = torch.empty(total, dtype=torch.int32, device=dev)
    dist_out = torch.empty(total, dtype=torch.int32, device=dev)
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.int32, device=dev)
    tuning = None
    if not args.no_autotune:  # launch parameters picked for this batch (results unaffected)
        tuning = u.autotune(d_shift, reps=1)
    for _ in range(args.warmup):
        cuts = u.decompose(betas, d_shift, center, dist_out)
    torch.cuda.synchronize()
    # ---- batched: one union decomposition (+ every member's cut count) per step
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    sts = []
    barrier(dist)
    torch.cuda.synchronize()
    with ClockSampler(local) as clocks:
        for i in range(args.steps):
            with torch.cuda.stream(stream):
                flush.fill_(i)
            ev[i][0].record(stream)
            cuts = u.decompose(betas, d_shift, center, dist_out)
            ev[i][1].record(stream)
            sts.append(u.stats())
        torch.cuda.synchronize()
    barrier(dist)
    ms = reduce_max(dist, sum(a.elapsed_time(b) for a, b in ev) / args.steps, dev)
    launches = sum(st["launches"] + st["cut_launches"] for st in sts)
    # ---- one at a time: ldd_decompose + ldd_cut_edges per member, same stream
    offs = u.offsets
    one_steps = max(1, min(args.steps, 3))
    e1 = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(one_steps)]
    one_cuts = []
    for i in range(one_steps):
        one_cuts = []
        with torch.cuda.stream(stream):
            flush.fill_(i)
        e1[i][0].record(stream)
        for s, mg in enumerate(members):
            lo, hi = offs[s], offs[s + 1]
            mg.decompose(betas[s], d_shift[lo:hi], center[lo:hi], dist_out[lo:hi])
            one_cuts.append(mg.cut_edges(center[lo:hi]))
        e1[i][1].record(stream)
    torch.cuda.synchronize()
    ms_one = reduce_max(dist, sum(a.elapsed_time(b) for a, b in e1) / one_steps, dev)
    one_c = center.cpu().numpy()
    one_d = dist_out.cpu().numpy()
    # ---- the batched outputs equal the one-at-a-time outputs (and cut counts)
    cuts = u.decompose(betas, d_shift, center, dist_out)
    same = (cuts == one_cuts and np.array_equal(center.cpu().numpy(), one_c)
            and np.array_equal(dist_out.cpu().numpy(), one_d))
    # ---- end to end with pinned host buffers
    h_shift = torch.from_numpy(np.concatenate(shifts)).pin_memory()
    h_c = torch.empty(total, dtype=torch.int32).pin_memory()
    h_d = torch.empty(total, dtype=torch.int32).pin_memory()
    u.decompose(betas, h_shift, h_c, h_d)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        u.decompose(betas, h_shift, h_c, h_d)
    e2e_s = reduce_max(dist, (time.perf_counter() - t0) / args.steps, dev)
    # ---- roofline of the BFS launch on the union: one regular (not replayed)
    # call with per-phase events, after the timed steps
    u.set_graph_replay(False)
    u.decompose(betas, d_shift, center, dist_out)
    st = u.stats()
    u.set_graph_replay(not args.no_replay)
    bfs_bytes = bfs_algorithmic_bytes(st)
    peak, peak_kind = measured_peak_hbm()
    bfs_ach = bfs_bytes / (st["ms_bfs"] * 1e-3) / 1e9
    # ---- CPU oracle on a bounded sample of members
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        import oracle

        t0 = time.perf_counter()
        done_m = done = 0
        for s in range(k):
            oc, od = oracle.oracle_ldd(Gs[s].row_ptr, Gs[s].col, shifts[s])
            assert np.array_equal(oc, one_c[offs[s]:offs[s + 1]]), f"member {s} differs from the oracle"
            oracle.oracle_cut_edges(Gs[s].row_ptr, Gs[s].col, oc)
            done += 1
            done_m += Gs[s].m
            if time.perf_counter() - t0 > 10.0:
                break
        t_cpu = time.perf_counter() - t0
        cpu = {"value": done / t_cpu, "unit": "decompositions/s", "cores": 1, "host_cores": os.cpu_count(), "kind": "oracle",
               "sample": f"the first {done} of {k} members, each checked equal to the GPU output",
               "gteps": done_m / t_cpu / 1e9}
    if rank == 0:
        clk = clocks.summary()
        line = {
            "metric": "LDD batched decompositions/s", "value": world * k / (ms * 1e-3),
            "unit": "decompositions/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
            "config": {"workload": args.workload, "batch": desc, "members": k,
                       "vertices": total, "m": m_total,
                       "step": "one ldd_union_decompose of the whole batch + every member's cut count",
                       "l2": "flushed between steps (inputs also exceed L2)",
                       "parallelism": f"replicas x{world}"},
            "gteps": world * m_total / (ms * 1e-3) / 1e9,
            "one_at_a_time": {"ms_per_batch": ms_one, "decompositions_per_s": world * k / (ms_one * 1e-3),
                              "speedup_of_batched": ms_one / ms, "api": "ldd_decompose + ldd_cut_edges per member"},
            "batched_equals_one_at_a_time": bool(same),
            "roofline": {"bound": "hbm", "kernel": "k_bfs", "achieved": bfs_ach, "peak": peak,
                         "unit": "GB/s", "frac": bfs_ach / peak, "traffic": None,
                         "peak_kind": f"of {peak_kind}", "algorithmic_bytes_per_launch": bfs_bytes,
                         "avg_launch_ms": st["ms_bfs"]},
            "cpu_baseline": cpu,
            "e2e": {"value": world * k / e2e_s, "unit": "decompositions/s",
                    "h2d_bytes_per_step": 8 * total, "d2h_bytes_per_step": 8 * total + 8 * k,
                    "ms_per_step": 1e3 * e2e_s, "api": "ldd_union_decompose (pinned host buffers)"},
            "gpu_launches": launches,
            "clocks": {"sm_mhz": clk["sm_mhz"], "sm_max_mhz": clk["sm_max_mhz"], "reasons": clk["reasons"]},
            "autotuned": tuning,
            "union": {"replayed_in_timed_steps": sts[-1]["replayed"],
                      "ms_replay": sts[-1]["ms_replay"], "rounds": st["rounds"], "pull_rounds": st["pull_rounds"], "A": st["max_floor_shift"],
                      "ms_rank": st["ms_rank"], "ms_bfs": st["ms_bfs"], "ms_finalize": st["ms_finalize"],
                      "ms_cut": st["ms_cut"], "ms_total": st["ms_total"], "exact_rank": st["exact_rank"],
                      "bfs_windows": st["bfs_windows"], "bfs_overflow": st["bfs_overflow"]},
            "host_s": {"generation": t_gen, "graph_and_union_creation": t_create},
            "create_graph": {"wall_ms": 1e3 * t_create,
                             "components_ms": sum(mg.stats()["ms_create_components"]
                                                  for mg in uniq.values()),
                             "note": "every member graph and the union, once per batch "
                                     "definition, outside the timed step"},
        }
    u.close()
    for mg in uniq.values():
        mg.close()
    return line if rank == 0 else None


# ----------------------------------------------------------------- serving
def serve_arm(args, dist):
    """A Poisson request stream replayed in real time against the batched
    server and, on the same stream, against one-at-a-time plain calls; at the
    workload's rate and at lower rates that the one-at-a-time server also
    sustains, so that its p50/p99 there are service latencies, not queue
    growth."""
    import numpy as np
    import torch

    import ldd_gen as gen
    import paper_1307_3692_gb300 as ldd

    world, rank, local = dist_env()
    dev = torch.device("cuda", local)
    spec = gen.SERVE_WORKLOADS[args.workload]
    t0 = time.perf_counter()
    Gs = [gen.rmat(sc) for sc in spec["rmat_scales"]] + [gen.grid2d(w, w) for w in spec["grids"]]
    names = [f"rmat{sc}" for sc in spec["rmat_scales"]] + [f"grid{w}x{w}" for w in spec["grids"]]
    gs = [ldd.LddGraph(torch.from_numpy(G.row_ptr).to(dev), torch.from_numpy(G.col).to(dev),
                       validate=False) for G in Gs]
    betas, S = spec["betas"], spec["seeds"]
    pool = {}
    for gi, G in enumerate(Gs):
        for bi, b in enumerate(betas):
            for si in range(S):
                pool[gi, bi, si] = torch.from_numpy(
                    gen.shifts(G.n, b, 1000 + 100 * gi + 10 * bi + si)).pin_memory()
    ring = 8  # output buffers per graph (results of a benchmark stream are not kept)
    outs = [[(torch.empty(G.n, dtype=torch.int32).pin_memory(),
              torch.empty(G.n, dtype=torch.int32).pin_memory()) for _ in range(ring)] for G in Gs]
    t_setup = time.perf_counter() - t0

    def replay(srv, reqs):
        check_every = max(1, len(reqs) // 16)
        # warm-up, untimed: one request per graph alone, then all of them at once,
        # so that first-use allocations and kernel loading of both the direct
        # and the union path happen before the stream starts
        for gi, G in enumerate(Gs):
            c, d = outs[gi][0]
            srv.wait(srv.submit(gs[gi], betas[0], pool[gi, 0, 0], c, d, np.zeros(1, np.int64)))
        warm = [srv.submit(gs[gi], betas[0], pool[gi, 0, 0], *outs[gi][1], np.zeros(1, np.int64))
                for gi in range(len(Gs))]
        for t in warm:
            srv.wait(t)
        tickets, checks, cuts = [], {}, []
        start = time.perf_counter()
        late = 0.0
        for i, (t_arr, gi, bi, si) in enumerate(reqs):
            while True:
                dt = t_arr - (time.perf_counter() - start)
                if dt <= 0:
                    late = max(late, -dt)
                    break
                if dt > 2e-4:
                    time.sleep(dt - 1e-4)
            if i % check_every == 0:
                c = np.empty(Gs[gi].n, np.int32)
                d = np.empty(Gs[gi].n, np.int32)
                checks[i] = (c, d)
            else:
                c, d = outs[gi][i % ring]
            cut = np.zeros(1, np.int64)
            cuts.append(cut)
            tickets.append(srv.submit(gs[gi], betas[bi], pool[gi, bi, si], c, d, cut))
        infos = [srv.wait(t) for t in tickets]
        return infos, checks, late

    def summarise(infos, late):
        lat = np.array([(x["end_us"] - x["submit_us"]) / 1e3 for x in infos])
        span = (max(x["end_us"] for x in infos) - min(x["submit_us"] for x in infos)) / 1e6
        bs = np.array([x["batch_size"] for x in infos])
        batches = {x["batch_id"]: x for x in infos}
        fill = np.array([x["batch_fill_us"] for x in batches.values()]) / 1e3
        run = np.array([x["batch_run_us"] for x in batches.values()]) / 1e3
        return {"requests": len(infos), "throughput_rps": len(infos) / span,
                "mean_batch_fill_ms": float(fill.mean()), "mean_batch_run_ms": float(run.mean()),
                # batches' device phases summed over the span: above 1 when the
                # workers' batches overlap on the device
                "batch_run_sum_over_span": float(run.sum() / 1e3 / span),
                "p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
                "mean_ms": float(lat.mean()), "max_ms": float(lat.max()),
                "batches": int(len(set(x["batch_id"] for x in infos))),
                "mean_batch_size": float(bs.mean()), "span_s": span,
                "max_submit_lag_ms": 1e3 * late}

    budget = spec["hbm_budget"]
    rates = sorted(set([r for r in (500.0, 1000.0) if r < spec["rate"]] + [spec["rate"]]))
    per_rate, mismatches, sampled = [], 0, 0
    clocks = ClockSampler(local)
    for rate in rates:
        reqs = gen.serve_requests(len(Gs), len(betas), S, rate, spec["seconds"],
                                  spec["master_seed"] + rank)
        srv = ldd.LddServer(budget, max_batch=args.max_batch, slots=2)
        if rate == spec["rate"]:
            with clocks:
                infos_b, checks_b, late_b = replay(srv, reqs)
        else:
            infos_b, checks_b, late_b = replay(srv, reqs)
        srv.close()
        one = ldd.LddServer(budget, max_batch=1, slots=1, one_at_a_time=True)
        infos_1, checks_1, late_1 = replay(one, reqs)
        one.close()
        batched, single = summarise(infos_b, late_b), summarise(infos_1, late_1)
        # mix check: sampled requests equal their results alone (and the other arm)
        for i, (c, d) in checks_b.items():
            _, gi, bi, si = reqs[i]
            ac = np.empty(Gs[gi].n, np.int32)
            ad = np.empty(Gs[gi].n, np.int32)
            gs[gi].decompose(betas[bi], pool[gi, bi, si], ac, ad)
            c1, d1 = checks_1[i]
            mismatches += int(not (np.array_equal(c, ac) and np.array_equal(d, ad)
                                   and np.array_equal(c1, ac) and np.array_equal(d1, ad)))
            sampled += 1
        sustained = single["throughput_rps"] >= 0.95 * rate
        per_rate.append({"rate_rps": rate, "requests": len(reqs), "batched": batched,
                         "one_at_a_time": single,
                         "one_at_a_time_sustains_rate": bool(sustained),
                         "p50_speedup": single["p50_ms"] / batched["p50_ms"],
                         "p99_speedup": single["p99_ms"] / batched["p99_ms"],
                         "throughput_speedup": batched["throughput_rps"] / single["throughput_rps"]})
    top = per_rate[-1]
    batched, single = top["batched"], top["one_at_a_time"]
    m_req = np.mean([Gs[gi].m for _, gi, _, _ in reqs])
    if rank == 0:
        clk = clocks.summary()
        line = {
            "metric": "LDD served decompositions/s", "value": world * batched["throughput_rps"],
            "unit": "decompositions/s", "n_gpus": world, "steps": 1, "warmup": len(Gs),
            "ms_per_step": 1e3 * batched["span_s"], "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "u64", "data": "synthetic",
            "config": {"workload": args.workload,
                       "graphs": names, "betas": list(betas), "shift_vectors_per_graph_beta": S,
                       "arrivals": f"Poisson, mean {spec['rate']:.0f}/s for {spec['seconds']} s "
                                   f"(seed {spec['master_seed']})",
                       "hbm_budget_bytes": budget, "slots": 2, "max_batch": args.max_batch,
                       "mean_edges_per_request": float(m_req),
                       "step": "the whole request stream, replayed in real time",
                       "parallelism": f"replicas x{world}"},
            "batched": batched, "one_at_a_time": single,
            "p99_speedup": single["p99_ms"] / batched["p99_ms"],
            "throughput_speedup": batched["throughput_rps"] / single["throughput_rps"],
            "by_rate": per_rate,
            "served_gteps": batched["throughput_rps"] * m_req / 1e9,
            "mix_check": {"sampled": sampled, "mismatches": mismatches,
                          "against": "ldd_decompose alone on the same graph and shifts, and "
                                     "the one-at-a-time server's result"},
            "roofline": None, "cpu_baseline": None,
            "e2e": {"value": world * batched["throughput_rps"], "unit": "decompositions/s",
                    "h2d_bytes_per_step": int(sum(8 * Gs[gi].n for _, gi, _, _ in reqs)),
                    "d2h_bytes_per_step": int(sum(8 * Gs[gi].n + 8 for _, gi, _, _ in reqs)),
                    "api": "ldd_server_submit / ldd_server_wait, pinned host buffers"},
            "gpu_launches": None,
            "clocks": {"sm_mhz": clk["sm_mhz"], "sm_max_mhz": clk["sm_max_mhz"],
                       "reasons": clk["reasons"]},
            "host_s": {"setup": t_setup},
            "create_graph": {"components_ms": sum(g.stats()["ms_create_components"] for g in gs),
                             "note": "the 15 resident graphs, once, before the stream starts"},
        }
    for g in gs:
        g.close()
    return line if rank == 0 else None


# ----------------------------------------------------------------- block decomposition
def blocks_arm(args, dist):
    """Blocks by repeated decomposition (ldd_block_decompose) of one graph per
    step, every block checked against the oracle's loop."""
    import numpy as np
    import torch

    import ldd_gen as gen
    import paper_1307_3692_gb300 as ldd

    world, rank, local = dist_env()
    dev = torch.device("cuda", local)
    spec = gen.BLOCK_WORKLOADS[args.workload]
    t0 = time.perf_counter()
    G = gen.make_graph(spec["graph"])
    k = spec["vectors"]
    shifts = [gen.shifts(G.n, spec["beta"], spec["first_seed"] + i) for i in range(k)]
    t_gen = time.perf_counter() - t0
    d_rp, d_col = torch.from_numpy(G.row_ptr).to(dev), torch.from_numpy(G.col).to(dev)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    g = ldd.LddGraph(d_rp, d_col, validate=False)
    create = create_info(g, time.perf_counter() - t0)
    del d_rp, d_col
    stream = torch.cuda.Stream(device=dev)
    g.set_stream(stream)
    d_sh = [torch.from_numpy(x).to(dev) for x in shifts]
    cs = [torch.empty(G.n, dtype=torch.int32, device=dev) for _ in range(k)]
    ds = [torch.empty(G.n, dtype=torch.int32, device=dev) for _ in range(k)]
    ab = torch.empty(G.nnz, dtype=torch.int32, device=dev)
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.int32, device=dev)
    betas = [spec["beta"]] * k
    for _ in range(args.warmup):
        g.block_decompose(betas, d_sh, cs, ds, ab)
    torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    sts = []
    barrier(dist)
    with ClockSampler(local) as clocks:
        for i in range(args.steps):
            with torch.cuda.stream(stream):
                flush.fill_(i)
            ev[i][0].record(stream)
            nb, rem = g.block_decompose(betas, d_sh, cs, ds, ab)
            ev[i][1].record(stream)
            sts.append(g.stats())
        torch.cuda.synchronize()
    barrier(dist)
    ms = reduce_max(dist, sum(a.elapsed_time(b) for a, b in ev) / args.steps, dev)
    st = sts[-1]
    # the residual passes' algorithmic bytes.  Count pass: per arc of G_i its
    # source, target, block stamp and two center gathers (20 B); write pass:
    # per kept arc the list entry, source, target and input id read, three
    # words written (28 B); G_0's per-vertex tables (counts, offsets, flags,
    # new ids: 28 B); later iterations' vertex passes cover only the few
    # vertices with a kept arc
    res_bytes = (20 * st["block_arcs_scanned"] + 28 * st["block_arcs_kept"] + 28 * G.n)
    peak, peak_kind = measured_peak_hbm()
    res_ach = res_bytes / (st["ms_block_residual"] * 1e-3) / 1e9 if st["ms_block_residual"] > 0 else 0.0
    parity = cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        import oracle

        t0 = time.perf_counter()
        oc, od, oab, orem = oracle.oracle_block_decompose(G.row_ptr, G.col, shifts)
        t_cpu = time.perf_counter() - t0
        bad = int((ab.cpu().numpy() != oab).sum())
        for i in range(len(oc)):
            bad += int((cs[i].cpu().numpy() != oc[i]).sum() + (ds[i].cpu().numpy() != od[i]).sum())
        parity = {"blocks": nb, "oracle_blocks": len(oc), "remaining_equal": rem == list(orem),
                  "mismatches": bad,
                  "method": "every arc's block and every iteration's centers and distances "
                            "against the oracle's loop"}
        assert bad == 0 and rem == list(orem) and nb == len(oc), parity
        cpu = {"value": G.m / t_cpu / 1e9, "unit": "GTEPS", "cores": 1,
               "host_cores": os.cpu_count(), "kind": "oracle", "seconds": t_cpu,
               "sample": f"one full block decomposition of {args.workload} ({len(oc)} iterations)"}
    g.close()
    if rank != 0:
        return None
    clk = clocks.summary()
    return {
        "metric": "LDD block decompositions/s", "value": world * 1e3 / ms,
        "unit": "block decompositions/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "u64", "data": "synthetic",
        "config": {"workload": args.workload,
                   "graph": f"R-MAT scale {spec['graph'][1]}, edge factor 16, seed 7",
                   "n": G.n, "m": G.m, "beta": spec["beta"], "shift_vectors": k,
                   "step": "one ldd_block_decompose: decompose, keep the cut edges, repeat until "
                           "none is left",
                   "l2": "flushed between steps", "parallelism": f"replicas x{world}"},
        "gteps": world * G.m / (ms * 1e-3) / 1e9,
        "blocks": nb, "remaining_edges": rem,
        "ms_residual_passes": st["ms_block_residual"],
        "ms_decompositions": st["ms_block_total"] - st["ms_block_residual"],
        "roofline": {"bound": "hbm", "kernel": "k_residual (count + write passes, scan, "
                                               "component tables)",
                     "achieved": res_ach, "peak": peak, "unit": "GB/s", "frac": res_ach / peak,
                     "traffic": None, "peak_kind": f"of {peak_kind}",
                     "algorithmic_bytes_per_call": res_bytes,
                     "share_of_step": st["ms_block_residual"] / max(st["ms_block_total"], 1e-9),
                     "note": "the decompositions of G_0, G_1, ... are the round-loop kernels of "
                             "the single-graph lines"},
        "cpu_baseline": cpu, "parity": parity,
        "e2e": None, "gpu_launches": None,
        "clocks": {"sm_mhz": clk["sm_mhz"], "sm_max_mhz": clk["sm_max_mhz"],
                   "reasons": clk["reasons"]},
        "host_s": {"generation": t_gen},
        "create_graph": create,
    }


# ----------------------------------------------------------------- Figure 1
def fig1_arm(args):
    """The paper's only experiment (Figure 1): a 1000 x 1000 grid decomposed at
    beta in {0.002, 0.005, 0.01, 0.02, 0.05, 0.1}.  The figure shows the
    pieces; this reports what it illustrates, per beta over a few shift
    seeds: pieces, radius, cut fraction against Corollary 3.5's 1 - e^-beta,
    delta_max against Lemma 3.2's H_n / beta, and the GPU time, with every
    labelling checked equal to the oracle's."""
    import numpy as np
    import torch

    import ldd_gen as gen
    import oracle
    import paper_1307_3692_gb300 as ldd

    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    G = gen.grid2d(1000, 1000)
    g = ldd.LddGraph(torch.from_numpy(G.row_ptr).to(dev), torch.from_numpy(G.col).to(dev),
                     validate=False)
    g.set_timing(True)
    c = torch.empty(G.n, dtype=torch.int32, device=dev)
    d = torch.empty(G.n, dtype=torch.int32, device=dev)
    H = float(np.sum(1.0 / np.arange(1, G.n + 1)))
    rows = []
    mismatches = 0
    seeds = range(1, 1 + max(1, args.steps))
    for beta in (0.002, 0.005, 0.01, 0.02, 0.05, 0.1):
        acc = {"pieces": [], "max_radius": [], "mean_radius": [], "cut_fraction": [],
               "delta_max": [], "ms": []}
        for seed in seeds:
            sh = gen.shifts(G.n, beta, seed)
            dsh = torch.from_numpy(sh).to(dev)
            g.decompose(beta, dsh, c, d)  # warm
            g.decompose(beta, dsh, c, d)
            ms = g.stats()["ms_total"]
            cut = g.cut_edges(c)
            gc, gd = c.cpu().numpy(), d.cpu().numpy()
            if not args.no_cpu_baseline:
                oc, od = oracle.oracle_ldd(G.row_ptr, G.col, sh)
                mismatches += int(not (np.array_equal(gc, oc) and np.array_equal(gd, od)))
            acc["pieces"].append(len(np.unique(gc)))
            acc["max_radius"].append(int(gd.max()))
            acc["mean_radius"].append(float(gd.mean()))
            acc["cut_fraction"].append(cut / G.m)
            acc["delta_max"].append(float(sh.max()))
            acc["ms"].append(ms)
        row = {"beta": beta} | {k: float(np.mean(v)) for k, v in acc.items()}
        row |= {"cut_bound_1_minus_exp": 1 - math.exp(-beta), "H_n_over_beta": H / beta,
                "gteps": G.m / (row["ms"] * 1e-3) / 1e9}
        rows.append(row)
    g.close()
    if rank == 0:
        print(json.dumps({
            "metric": "LDD Figure 1 sweep", "value": float(np.mean([r["gteps"] for r in rows])),
            "unit": "GTEPS", "n_gpus": 1, "steps": len(seeds), "warmup": 1,
            "higher_is_better": True, "data": "synthetic", "dtype": "u64",
            "config": {"workload": "fig1", "graph": "2D 4-neighbour grid 1000x1000",
                       "seeds": list(seeds)},
            "rows": rows, "oracle_mismatches": None if args.no_cpu_baseline else mismatches}),
            flush=True)
    return 0


# Lines nested in the default run's output, after the headline: every other
# configuration of the method (workload, arm, most timed steps).
EXTRAS = [
    ("grid2d_256", "single", 20),
    ("grid3d_256", "single", 10),
    ("rmat20_seeds_64", "batch", 5),
    ("rgg_batch_1024", "batch", 3),
    ("rmat20_blocks", "blocks", 5),
    ("serve_mix", "serve", 1),
]


def run_arm(kind, args, dist):
    return {"single": our_arm, "batch": batch_arm, "serve": serve_arm,
            "blocks": blocks_arm}[kind](args, dist)


CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
            "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "roofline",
            "cpu_baseline", "e2e", "gpu_launches", "clocks", "kernel_source_sha")


def short(line, nested):
    """The default run's printed line: a reader that keeps the last few thousand
    characters of the output gets all of it.  The whole lines go to stderr."""
    out = {k: line[k] for k in CONTRACT if k in line}
    out["workloads"] = {name: {k: x.get(k) for k in ("value", "unit", "ms_per_step")}
                        for name, x in nested.items()}
    return out


def main(argv=None):
    ap = argparse.ArgumentParser(description=__doc__.split("\n")[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", default="rmat22")
    ap.add_argument("--single", action="store_true",
                    help="only the named workload's line (the default R-MAT 22 run also nests "
                         "a line for every other configuration)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--max-batch", type=int, default=256,
                    help="serving: most requests per batch")
    ap.add_argument("--no-autotune", action="store_true",
                    help="batched workloads: keep the default launch parameters")
    ap.add_argument("--no-replay", action="store_true",
                    help="batched workloads: run the regular path instead of the captured CUDA graph")
    args = ap.parse_args(argv)
    args.warmup = max(args.warmup, 3)  # at least three untimed warm-up steps
    import ldd_gen

    kinds = {name: "single" for name in ldd_gen.WORKLOADS}
    kinds.update({name: "batch" for name in ldd_gen.BATCH_WORKLOADS})
    kinds.update({name: "serve" for name in ldd_gen.SERVE_WORKLOADS})
    kinds.update({name: "blocks" for name in ldd_gen.BLOCK_WORKLOADS})
    kinds["fig1"] = "fig1"
    if args.workload not in kinds:
        ap.error(f"unknown workload {args.workload}")
    kind = kinds[args.workload]
    if args.impl == "reference":
        if kind == "single":
            return reference_arm(args)
        why = {"fig1": "the Figure 1 sweep checks every labelling against the oracle itself",
               "serve": "the serving workload has no reference arm; its line compares against "
                        "one-at-a-time plain calls",
               "batch": "the batched workloads have no reference arm; their line carries the "
                        "oracle's sample as cpu_baseline",
               "blocks": "the block decomposition's line carries the oracle's loop as "
                         "cpu_baseline"}[kind]
        print(json.dumps({"impl": "reference", "unavailable": why}), flush=True)
        return 0
    if kind == "fig1":
        return fig1_arm(args)
    import torch

    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    dist = init_dist(world, "nccl")
    line = run_arm(kind, args, dist)
    if args.workload == "rmat22" and not args.single:
        nested = {}
        for name, sub_kind, max_steps in EXTRAS:
            sub = argparse.Namespace(**vars(args))
            sub.workload = name
            sub.steps = max(1, min(args.steps, max_steps))
            torch.cuda.empty_cache()
            nested[name] = run_arm(sub_kind, sub, dist)
        if rank == 0:
            for name, x in ((args.workload, line), *nested.items()):
                print(json.dumps({name: x}), file=sys.stderr, flush=True)
            line = short(line, nested)
    if rank == 0 and line is not None:
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
