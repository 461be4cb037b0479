"""Benchmark of the GAS superstep engine: PageRank on R-MAT scale 22.

One step = one complete PageRank run through the C-ABI (gxp_begin + 20
supersteps of MSGGen/MSGMerge/MSGApply) on 4,194,304 vertices and 67,108,864
edges, d = 0.85. The metric is GTEPS (edges scanned per second over all
supersteps) and the HBM-roofline fraction of the superstep kernel.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gxp|reference]

--impl reference times the CPU oracle (the plain fp64 C loop) on a bounded
sample of the same workload: each step is one full-graph PageRank superstep.
Under torchrun (N > 1) every rank runs an independent replica on its own GPU
(no data-path collective); rank 0 prints one JSON line.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

REPO = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, REPO)

from paper_2203_13005_gb300 import synth  # noqa: E402

METRIC = "GTEPS & % HBM roofline per GAS superstep"
# superstep directions of the min-label runs (gxp_direction)
DIRECTIONS = {"auto": 0, "pull": 1, "push": 2}
ITERS = 20
DAMPING = 0.85
WL = synth.PAGERANK_RMAT22
PROFILE = os.path.join(REPO, "profiles", "superstep_pagerank_rmat22.txt")
PROFILE_CC = os.path.join(REPO, "profiles", "superstep_cc_er24_8parts.txt")
KERNEL_SRC = os.path.join(REPO, "paper_2203_13005_gb300", "csrc", "sweep.cu")     # one partition
KERNEL_SRC_CC = os.path.join(REPO, "paper_2203_13005_gb300", "csrc", "sell.cu")   # several


def algorithmic_bytes(n_vertices: int, n_edges: int) -> int:
    """Bytes one PageRank superstep must move at minimum: per edge the source
    index (4) and the gathered contribution (4); per vertex col_ptr (4),
    out-degree (4), new rank (4), new contribution (4): 604.0 MB at R-MAT 22."""
    return 8 * n_edges + 16 * n_vertices


def algorithmic_bytes_with_old_rank(n_vertices: int, n_edges: int) -> int:
    """The same plus the old rank (4 B per vertex), which the kernel also reads
    to form the exact sum of |r_new - r_old| (the convergence sum)."""
    return 8 * n_edges + 20 * n_vertices


def measured_peaks() -> dict:
    p = os.path.join(REPO, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return {"hbm_gbs": float(d["hbm_gbs"]), "source": "measured"}
    return {"hbm_gbs": 6800.0, "source": "fallback"}


def profiled_traffic(profile=None, kernel_src=None):
    """Per-launch DRAM bytes from a committed ncu summary (the PageRank one by
    default), if it was taken on the current kernel source (its sha256 is
    recorded there); else None."""
    profile = profile or PROFILE
    if not os.path.exists(profile):
        return None
    kv = {}
    for ln in open(profile):
        if ":" in ln and not ln.startswith("#"):
            k, v = ln.split(":", 1)
            kv[k.strip()] = v.strip()
    sha = hashlib.sha256(open(kernel_src or KERNEL_SRC, "rb").read()).hexdigest()
    if kv.get("kernel_source_sha256") != sha or "dram_bytes_per_launch" not in kv:
        return None
    return float(kv["dram_bytes_per_launch"])


class ClockSampler:
    """nvidia-smi clock/throttle samples during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *a):
        self.lines = []
        if self.proc is not None:
            time.sleep(0.2)
            self.proc.terminate()
            try:
                out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                out, _ = self.proc.communicate()
            self.lines = [ln for ln in out.splitlines() if ln.strip()]

    def summary(self) -> dict:
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in getattr(self, "lines", []):
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for nm, val in zip(names, f[5:9]):
                if val.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx,
                "reasons": sorted(reasons), "samples": len(sm)}


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def run_reference(args, world, rank):
    """The oracle as it stands, single-threaded fp64 C, on host cores."""
    if rank != 0:
        return
    import oracle
    src, dst, _ = WL.edges()
    n, m = WL.n_vertices, WL.n_edges
    outdeg_unused = None  # noqa: F841  (the oracle counts out-degrees itself)
    r = np.full(n, 1.0 / n)
    for _ in range(args.warmup):
        r, _, _ = oracle.pagerank_step(n, src, dst, r, DAMPING)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        r, _, _ = oracle.pagerank_step(n, src, dst, r, DAMPING)
    dt = time.perf_counter() - t0
    gteps = args.steps * m / dt / 1e9
    line = {
        "impl": "reference", "metric": METRIC, "value": gteps, "unit": "GTEPS", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt / args.steps * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": WL.name, "vertices": n, "edges": m, "damping": DAMPING,
                   "step": "one PageRank superstep over the full graph (oracle)"},
        "cpu_baseline": {"value": gteps, "unit": "GTEPS", "cores": 1, "kind": "oracle",
                         "sample": f"{args.steps} full-graph fp64 supersteps of {WL.name}"},
        "e2e": {"value": gteps, "unit": "GTEPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0,
    }
    print(json.dumps(line), flush=True)


def host_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


def cpu_baseline(src, dst, n, m):
    """Oracle PageRank on this host: one whole step of the workload (its 20
    full-graph supersteps, about 10 s of single-threaded CPU work)."""
    import oracle
    k = ITERS
    t0 = time.perf_counter()
    oracle.pagerank(n, src, dst, DAMPING, k)
    dt = time.perf_counter() - t0
    return {"value": k * m / dt / 1e9, "unit": "GTEPS", "cores": 1, "host_cores": host_cores(), "kind": "oracle",
            "sample": f"{k} fp64 supersteps of {WL.name} (single thread, incl. its out-degree pass)"}


def cpu_all_cores_pagerank(src, dst, n, m):
    """The same 20 PageRank supersteps (fp64, pulled by destination over a CSC)
    on every host core with OpenMP: a parallel CPU baseline, not the oracle.
    The CSC is built before the timed region."""
    from oracle import cpu_baselines as cb
    cores = cb.set_threads(host_cores())
    col_ptr, csrc, _ = cb.csc(n, src, dst)
    outdeg = np.bincount(src, minlength=n).astype(np.uint32)
    t0 = time.perf_counter()
    cb.pagerank_pull(n, col_ptr, csrc, outdeg, DAMPING, ITERS)
    dt = time.perf_counter() - t0
    return {"value": ITERS * m / dt / 1e9, "unit": "GTEPS", "cores": cores, "host_cores": host_cores(),
            "kind": "openmp pull by destination (fp64)",
            "sample": f"{ITERS} supersteps of {WL.name}, CSC built outside the timed region"}


def run_msssp(args):
    """Batched 64-source SSSP on R-MAT scale 24 with streamed edge blocks: the
    pipeline shuffle with the autotuned block size, against a fixed block size,
    no pipelining, and resident edges (the paper's pipeline-shuffle experiment
    restated on one GPU)."""
    import torch
    from paper_2203_13005_gb300 import gxp
    wl = synth.MSSSP_RMAT24
    src, dst, w = wl.edges()
    n, m = wl.n_vertices, wl.n_edges
    sources = synth.sources_with_out_edges(n, src, 64, wl.seed)
    ctx = gxp.Context(0)
    ctx.create_graph(n, 1)
    ctx.load_coo(src, dst, w)
    del src, dst, w
    dist = torch.empty((n, 64), dtype=torch.int32, device="cuda")
    runs = {}
    _, rep = ctx.sssp_batch(sources, out=dist, streamed=True, block_edges=0, use_graph=True)
    tuned = rep["block_edges"]
    runs["streamed_autotuned"] = rep
    for _ in range(max(1, args.steps)):
        _, rep = ctx.sssp_batch(sources, out=dist, streamed=True, block_edges=tuned, use_graph=True)
        runs["streamed_autotuned"] = rep if rep["ms_total"] < runs["streamed_autotuned"]["ms_total"] else runs["streamed_autotuned"]
    _, runs["streamed_fixed_1_8"] = ctx.sssp_batch(sources, out=dist, streamed=True, block_edges=m // 8, use_graph=True)
    _, runs["streamed_unpipelined"] = ctx.sssp_batch(sources, out=dist, streamed=True, pipelined=False,
                                                     block_edges=tuned, use_graph=True)
    _, runs["resident"] = ctx.sssp_batch(sources, out=dist)
    best = runs["streamed_autotuned"]
    sec = best["ms_total"] * 1e-3
    # roofline of k_msssp on the resident run (algorithmic bytes: 8 B per
    # scanned edge, 256 B per active edge's row gather, 524 B per vertex per
    # superstep), and the host link of the streamed run against a pinned copy
    peaks = measured_peaks()
    res = runs["resident"]
    res_bytes = 8 * m * res["supersteps"] + 256 * res["active_edges"] + 524 * n * res["supersteps"]
    res_gbs = res_bytes / (res["ms_total"] * 1e-3) / 1e9
    esize = 4 if wl.w_hi < 256 and n <= (1 << 24) else 8   # packed (weight << 24 | source) edges
    h2d = esize * m * best["supersteps"]
    line_gbs = pinned_h2d_gbs(torch)
    line = {
        "metric": METRIC, "value": best["supersteps"] * m / sec / 1e9, "unit": "GTEPS",
        "source_gteps": 64 * best["supersteps"] * m / sec / 1e9, "n_gpus": 1, "steps": args.steps,
        "warmup": 1, "ms_per_step": best["ms_total"], "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "u32", "data": "synthetic",
        "config": {"workload": wl.name, "vertices": n, "edges": m, "sources": 64,
                   "step": "one batched run to convergence, edges streamed from pinned host memory"},
        "runs": {k: {kk: (round(vv, 9) if isinstance(vv, float) else vv) for kk, vv in v.items()}
                 for k, v in runs.items()},
        "roofline": {"bound": "hbm", "achieved": res_gbs, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                     "frac": res_gbs / peaks["hbm_gbs"], "traffic": None, "peak_source": peaks["source"],
                     "kernel": "k_msssp (resident run)", "algorithmic_bytes_per_run": res_bytes,
                     "active_edges": res["active_edges"], "supersteps": res["supersteps"]},
        "link": {"h2d_bytes_per_superstep": esize * m, "achieved_gbs": h2d / sec / 1e9,
                 "pinned_copy_gbs": line_gbs, "frac": h2d / sec / 1e9 / line_gbs if line_gbs else None},
    }
    print(json.dumps(line), flush=True)
    ctx.close()


def pinned_h2d_gbs(torch) -> float:
    """Host-to-device bandwidth of one 1 GiB copy from pinned memory (best of 3)."""
    h = torch.empty(1 << 30, dtype=torch.uint8).pin_memory()
    d = torch.empty(1 << 30, dtype=torch.uint8, device="cuda")
    best = None
    for _ in range(3):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        d.copy_(h, non_blocking=True)
        b.record()
        torch.cuda.synchronize()
        t = a.elapsed_time(b) * 1e-3
        best = t if best is None else min(best, t)
    del h, d
    return (1 << 30) / best / 1e9


def run_sssp(args):
    """SSSP (Bellman-Ford, min merge) on R-MAT scale 16 (or 22) from source 0
    to convergence: supersteps are enqueued in chunks with one host read of
    their changed counts per chunk (gxp_run), each superstep pulling or
    pushing as --direction says. GTEPS = supersteps x edges / run time; the
    roofline is taken per pull superstep over a full sweep (at scale 16 the
    whole 13 MB working set is L2-resident, so it is quoted against HBM only
    for comparison)."""
    import torch
    from paper_2203_13005_gb300 import gxp
    wl = synth.SSSP_RMAT22 if args.workload == synth.SSSP_RMAT22.name else synth.SSSP_RMAT16
    src, dst, w = wl.edges()
    n, m = wl.n_vertices, wl.n_edges
    stream = torch.cuda.Stream()
    direction = DIRECTIONS[args.direction]
    ctx = gxp.Context(0, direction=direction, push_div=args.push_div)
    ctx.set_stream(stream.cuda_stream)
    ctx.create_graph(n, 1)
    ctx.load_coo(src, dst, w)
    for _ in range(args.warmup):
        steps = ctx.run(gxp.GXP_ALGO_SSSP, 0)
    reps = max(args.steps, 10)
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(0) as clk:
        torch.cuda.synchronize()
        t0.record(stream)
        for _ in range(reps):
            steps = ctx.run(gxp.GXP_ALGO_SSSP, 0)
        t1.record(stream)
        torch.cuda.synchronize()
    ms = t0.elapsed_time(t1) / reps
    st = ctx.stats()
    g, mm, a = gxp.TEMPLATES[gxp.GXP_ALGO_SSSP]

    def superstep_us(c):
        # one run's supersteps, each bracketed by events on the context's stream
        c.begin(gxp.GXP_ALGO_SSSP, 0)
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
        for b, e in evs:
            b.record(stream)
            c.lib.gxp_superstep(c.h, gxp.GXP_ALGO_SSSP, g, mm, a, None)
            e.record(stream)
        torch.cuda.synchronize()
        return [b.elapsed_time(e) * 1e3 for b, e in evs]

    per_step_us = superstep_us(ctx)
    # the pull kernel's roofline: every superstep in pull direction
    cp = gxp.Context(0, direction=gxp.GXP_DIR_PULL)
    cp.set_stream(stream.cuda_stream)
    cp.create_graph(n, 1)
    cp.load_coo(src, dst, w)
    superstep_us(cp)
    k_us = statistics.mean(superstep_us(cp))
    cp.close()
    bytes_sweep = 12 * m + 12 * n + n // 4   # src + w + gathered value per edge; col_ptr, d read, d write, bitmap
    # end to end through the public API with host buffers: weighted CSC from
    # pinned host memory -> load (device build) -> run -> distances back into
    # pinned host memory
    order = np.argsort(dst, kind="stable")
    col_ptr = torch.zeros(n + 1, dtype=torch.int64).pin_memory()
    np.cumsum(np.bincount(dst, minlength=n), out=col_ptr.numpy()[1:])
    csc_src = torch.from_numpy(np.ascontiguousarray(src[order]).view(np.int32)).pin_memory()
    csc_w = torch.from_numpy(np.ascontiguousarray(w[order]).view(np.int32)).pin_memory()
    del order
    out = torch.empty(n, dtype=torch.int32).pin_memory()
    e2e = []
    c2 = gxp.Context(0, direction=direction, push_div=args.push_div)
    c2.set_stream(stream.cuda_stream)
    for i in range(4):
        torch.cuda.synchronize()
        c0 = time.perf_counter()
        c2.create_graph(n, 1)
        c2.load_partition(0, gxp.GXP_FMT_CSC, m, col_ptr, csc_src, csc_w)
        c2.run(gxp.GXP_ALGO_SSSP, 0)
        c2.values(out=out)
        torch.cuda.synchronize()
        if i:
            e2e.append(time.perf_counter() - c0)
    c2.close()
    e2e_s = statistics.median(e2e)
    peaks = measured_peaks()
    cpu = {} if args.no_cpu_baseline else cpu_sssp_baselines(wl, src, dst, w, n, m)
    line = {
        "metric": METRIC, "value": steps * m / (ms * 1e-3) / 1e9, "unit": "GTEPS", "n_gpus": 1, "steps": reps,
        "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "u32", "data": "synthetic",
        "config": {"workload": wl.name, "vertices": n, "edges": m, "source": 0, "supersteps": steps,
                   "step": (f"one gxp_run to convergence: {st['persistent_launches']} persistent "
                            "launch(es), grid barrier between supersteps"),
                   "value": "supersteps x edges / run time (the Jacobi sweeps the run stands for)",
                   "l2": (f"{bytes_sweep / 1e6:.0f} MB working set: "
                          + ("L2-resident" if bytes_sweep < 129e6 else "larger than L2")),
                   "direction": args.direction,
                   "push_div": args.push_div or 8, "push_supersteps": st["push_supersteps"],
                   "edges_relaxed_per_run": st["edges_scanned"],
                   "superstep_us": [round(x, 2) for x in per_step_us],
                   "graph500_gteps": m / (ms * 1e-3) / 1e9},
        "roofline": {"bound": "hbm", "achieved": bytes_sweep / (k_us * 1e-6) / 1e9, "peak": peaks["hbm_gbs"],
                     "unit": "GB/s", "frac": bytes_sweep / (k_us * 1e-6) / 1e9 / peaks["hbm_gbs"], "traffic": None,
                     "peak_source": peaks["source"], "kernel": "k_sweep<SSSP>", "avg_launch_us": k_us,
                     "algorithmic_bytes_per_launch": bytes_sweep},
        "e2e": {"value": steps * m / e2e_s / 1e9, "unit": "GTEPS", "h2d_bytes_per_step": 8 * (n + 1) + 8 * m,
                "d2h_bytes_per_step": 4 * n, "ms_per_step": e2e_s * 1e3},
        # per run: the initial state, then the persistent kernel's launches
        "gpu_launches": reps * (1 + st["persistent_launches"]),
        "clocks": clk.summary(),
    }
    line.update(cpu)
    print(json.dumps(line), flush=True)
    ctx.close()


def cpu_sssp_baselines(wl, src, dst, w, n, m) -> dict:
    """SSSP from vertex 0 on the host: the oracle's Jacobi run (one core), the
    same supersteps pulled by destination on every core (OpenMP), and a
    binary-heap Dijkstra (one core). Each is checked against the oracle's
    distances; the CSC / CSR are built before the timed regions."""
    import oracle
    from oracle import cpu_baselines as cb
    t0 = time.perf_counter()
    d_ref, steps, _ = oracle.sssp(n, src, dst, w, 0)
    t_orc = time.perf_counter() - t0
    cores = cb.set_threads(host_cores())
    cp, cs, cw = cb.csc(n, src, dst, w)
    d0 = np.full(n, 0xFFFFFFFF, np.uint32)
    d0[0] = 0
    t0 = time.perf_counter()
    d_all, steps_all = cb.minlabel_pull(n, cp, cs, cw, d0)
    t_all = time.perf_counter() - t0
    rp, rd, rw = cb.csr(n, src, dst, w)
    t0 = time.perf_counter()
    d_dij = cb.dijkstra(n, rp, rd, rw, 0)
    t_dij = time.perf_counter() - t0
    if not (np.array_equal(d_all, d_ref) and np.array_equal(d_dij, d_ref) and steps_all == steps):
        raise RuntimeError("a CPU baseline disagrees with the oracle")
    hc = host_cores()
    return {
        "cpu_baseline": {"value": steps * m / t_orc / 1e9, "unit": "GTEPS", "cores": 1, "host_cores": hc,
                         "kind": "oracle", "sample": f"one whole run of {wl.name} ({steps} Jacobi supersteps)"},
        "cpu_baseline_all_cores": {"value": steps * m / t_all / 1e9, "unit": "GTEPS", "cores": cores,
                                   "host_cores": hc, "kind": "openmp pull by destination",
                                   "sample": f"one whole run of {wl.name}, CSC built outside the timed region"},
        "cpu_baseline_dijkstra": {"value": m / t_dij / 1e9, "unit": "GTEPS (edges / run time)", "cores": 1,
                                  "host_cores": hc, "kind": "binary-heap Dijkstra", "ms": t_dij * 1e3,
                                  "sample": f"source 0 of {wl.name}, CSR built outside the timed region"},
    }


def cpu_cc_baselines(wl, src, dst, n, m) -> dict:
    """Connected components on the host: one superstep of the oracle (one core,
    a bounded sample of the run), one superstep pulled by destination on every
    core, and the whole answer by union-find (one core)."""
    import oracle
    from oracle import cpu_baselines as cb
    lab0 = np.arange(n, dtype=np.uint32)
    t0 = time.perf_counter()
    l1, _ = oracle.cc_step(n, src, dst, lab0)
    t_orc = time.perf_counter() - t0
    cores = cb.set_threads(host_cores())
    cp, cs, _ = cb.csc(n, src, dst)
    t0 = time.perf_counter()
    l1_all, _ = cb.minlabel_pull(n, cp, cs, None, lab0, max_steps=1)
    t_all = time.perf_counter() - t0
    del cp, cs
    t0 = time.perf_counter()
    uf = cb.union_find(n, src, dst)
    t_uf = time.perf_counter() - t0
    if not np.array_equal(l1_all, l1):
        raise RuntimeError("the all-cores superstep disagrees with the oracle")
    hc = host_cores()
    return {
        "cpu_baseline": {"value": m / t_orc / 1e9, "unit": "GTEPS", "cores": 1, "host_cores": hc, "kind": "oracle",
                         "sample": f"the first superstep of {wl.name} (all edges)"},
        "cpu_baseline_all_cores": {"value": m / t_all / 1e9, "unit": "GTEPS", "cores": cores, "host_cores": hc,
                                   "kind": "openmp pull by destination",
                                   "sample": f"the first superstep of {wl.name}, CSC built outside the timed region"},
        "cpu_baseline_union_find": {"value": m / t_uf / 1e9, "unit": "GTEPS (edges / run time)", "cores": 1,
                                    "host_cores": hc, "kind": "union-find (path halving)", "ms": t_uf * 1e3,
                                    "sample": f"all components of {wl.name}"},
    }, uf


def sweep_launch_us(kernel_ms, reads_every_edge):
    """Average launch time (us) of the supersteps that read every edge, and
    their count: the roofline's launches are the pull supersteps, since a
    push superstep reads only its frontier's out-edges. With none, all."""
    sel = [k for k, f in zip(kernel_ms, reads_every_edge) if f]
    if not sel:
        sel = list(kernel_ms)
    return statistics.mean(sel) * 1e3, len(sel)


def run_cc(args):
    """Connected components (min-label propagation) on the Erdős–Rényi graph with
    2^24 vertices and 2^28 directed edges in 8 partitions with sync caching and
    skipping: per-superstep GTEPS, exchange statistics, roofline of the kernel."""
    import torch
    from paper_2203_13005_gb300 import gxp
    wl = synth.CC_ER24_P8 if args.cc_scale == 24 else synth.CC_ER24_P8.scaled(args.cc_scale)
    src, dst, _ = wl.edges()
    n, m = wl.n_vertices, wl.n_edges
    cpu, uf = ({}, None) if args.no_cpu_baseline else cpu_cc_baselines(wl, src, dst, n, m)
    ctx = gxp.Context(0, cache_slots=args.cache_slots)
    ctx.create_graph(n, wl.parts)
    ctx.load_coo(src, dst)
    del src, dst
    times = []
    steps = 0
    with ClockSampler(0) as clk:
        for r in range(max(2, args.steps)):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            steps = ctx.run(gxp.GXP_ALGO_CC)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
    st = ctx.stats()
    if uf is not None and not np.array_equal(ctx.values(), uf):
        raise RuntimeError("GPU components differ from union-find")
    sec = min(times[1:]) if len(times) > 1 else times[0]
    # the superstep kernel alone (k_sell<CC>, events around it on the context's
    # stream) and the whole superstep with its exchange, superstep by superstep
    ctx.begin(gxp.GXP_ALGO_CC)
    k_ms, s_ms, sweep = [], [], []
    for _ in range(steps):
        e0 = ctx.stats()["edges_scanned"]
        ctx.superstep()
        sx = ctx.stats()
        k_ms.append(sx["last_kernel_ms"])
        s_ms.append(sx["last_superstep_ms"])
        sweep.append(sx["edges_scanned"] - e0 == m)
    k_us, n_sweep = sweep_launch_us(k_ms, sweep)
    bytes_sweep = 8 * m + 12 * n + n // 4   # source id + gathered label per edge; col_ptr, old, new, bitmap
    peaks = measured_peaks()
    line = {
        "metric": METRIC, "value": steps * m / sec / 1e9, "unit": "GTEPS", "n_gpus": 1,
        "steps": len(times) - 1, "warmup": 1, "ms_per_step": sec * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
        "config": {"workload": wl.name, "vertices": n, "edges": m, "partitions": wl.parts,
                   "cache_slots": args.cache_slots,
                   "step": "one run to convergence incl. per-chunk host checks",
                   "l2": "inputs larger than L2: 1 GiB of edge indices per superstep vs 129 MB L2"},
        "supersteps": steps, "syncs_done": st["syncs_done"], "syncs_skipped": st["syncs_skipped"],
        "sync_pairs": st["sync_pairs"], "cache_downloads": st["cache_downloads"],
        "superstep_kernel_us": [round(x * 1e3, 1) for x in k_ms],
        "superstep_reads_every_edge": sweep, "push_supersteps": st["push_supersteps"],
        "superstep_with_sync_us": [round(x * 1e3, 1) for x in s_ms],
        "roofline": {"bound": "hbm", "achieved": bytes_sweep / (k_us * 1e-6) / 1e9, "peak": peaks["hbm_gbs"],
                     "unit": "GB/s", "frac": bytes_sweep / (k_us * 1e-6) / 1e9 / peaks["hbm_gbs"],
                     "traffic": profiled_traffic(PROFILE_CC, KERNEL_SRC_CC) if args.cc_scale == 24 else None,
                     "peak_source": peaks["source"], "kernel": "k_sell<CC>",
                     "avg_launch_us": k_us, "algorithmic_bytes_per_launch": bytes_sweep,
                     "launches_averaged": f"the {n_sweep} pull supersteps (every edge read) "
                                          f"of {steps}"},
        "gpu_launches": None, "clocks": clk.summary(),
    }
    line.update(cpu)
    print(json.dumps(line), flush=True)
    ctx.close()


def run_sync_skip(args):
    """SSSP (Bellman-Ford) from vertex 0 on the clustered graph (2^24
    vertices, 2^28 directed edges, 8 communities on the 8 partitions, one pair
    in 10^5 crossing): the sync-skipping experiment. Reports the exchanges
    done and skipped, the pairs moved, and GTEPS over the run."""
    import torch
    from paper_2203_13005_gb300 import gxp
    wl = synth.SSSP_CLUSTERED24_P8
    src, dst, w = wl.edges()
    n, m = wl.n_vertices, wl.n_edges
    ctx = gxp.Context(0)
    ctx.create_graph(n, wl.parts)
    ctx.load_coo(src, dst, w)
    del src, dst, w
    times = []
    steps = 0
    with ClockSampler(0) as clk:
        for r in range(max(2, args.steps)):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            steps = ctx.run(gxp.GXP_ALGO_SSSP, 0)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
    st = ctx.stats()
    sec = min(times[1:]) if len(times) > 1 else times[0]
    line = {
        "metric": METRIC, "value": steps * m / sec / 1e9, "unit": "GTEPS", "n_gpus": 1,
        "steps": len(times) - 1, "warmup": 1, "ms_per_step": sec * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
        "config": {"workload": wl.name, "vertices": n, "edges": m, "partitions": wl.parts,
                   "p_cross": wl.p_cross, "source": 0,
                   "step": "one SSSP run to convergence incl. per-chunk host checks"},
        "supersteps": steps, "syncs_done": st["syncs_done"], "syncs_skipped": st["syncs_skipped"],
        "skipped_fraction": st["syncs_skipped"] / max(1, steps), "sync_pairs": st["sync_pairs"],
        "clocks": clk.summary(),
    }
    print(json.dumps(line), flush=True)
    ctx.close()


def run_lp(args):
    """Label propagation (mode merge, ties to the smallest label, at most 15
    supersteps as in the paper's LP runs) on the Erdős–Rényi graph of the CC
    workload (2^24 vertices, 2^28 directed edges) in 8 partitions with sync
    caching and skipping. GTEPS = supersteps x edges / run time; the roofline
    counts 8 B per edge (source id, gathered label) and 40 B per row (its
    descriptor, old and new label) over the run's supersteps."""
    import torch
    from paper_2203_13005_gb300 import gxp
    if args.lp_graph == "rmat":
        # a power-law graph: the PageRank R-MAT recipe at --lp-scale, stored
        # in both directions (rows of every in-degree class, hub rows included)
        wl = synth.PAGERANK_RMAT22.scaled(args.lp_scale)
        s0, d0, _ = wl.edges()
        src, dst = np.concatenate([s0, d0]), np.concatenate([d0, s0])
        del s0, d0
    else:
        wl = synth.CC_ER24_P8 if args.lp_scale == 24 else synth.CC_ER24_P8.scaled(args.lp_scale)
        src, dst, _ = wl.edges()
    n, m = wl.n_vertices, len(src)
    parts = args.lp_parts
    ctx = gxp.Context(0)
    ctx.create_graph(n, parts)
    ctx.load_coo(src, dst)
    del src, dst
    cap = 15
    times = []
    steps = 0
    with ClockSampler(0) as clk:
        for r in range(max(2, args.steps)):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            steps = ctx.run(gxp.GXP_ALGO_LP, max_steps=cap)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
    st = ctx.stats()
    sec = min(times[1:]) if len(times) > 1 else times[0]
    # per-superstep device time (events around each superstep incl. its sync)
    stream = torch.cuda.Stream()
    ctx.set_stream(stream.cuda_stream)
    ctx.begin(gxp.GXP_ALGO_LP)
    g, mm, a = gxp.TEMPLATES[gxp.GXP_ALGO_LP]
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    for b, e in evs:
        b.record(stream)
        ctx.lib.gxp_superstep(ctx.h, gxp.GXP_ALGO_LP, g, mm, a, None)
        e.record(stream)
    torch.cuda.synchronize()
    step_us = [b.elapsed_time(e) * 1e3 for b, e in evs]
    k_us = statistics.mean(step_us)
    bytes_step = 8 * m + 40 * n
    peaks = measured_peaks()
    line = {
        "metric": METRIC, "value": steps * m / sec / 1e9, "unit": "GTEPS", "n_gpus": 1,
        "steps": len(times) - 1, "warmup": 1, "ms_per_step": sec * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
        "config": {"workload": f"lp_{args.lp_graph}{wl.scale}_{parts}parts", "vertices": n, "edges": m,
                   "partitions": parts,
                   "max_supersteps": cap, "step": "one LP run (to a quiet superstep or the cap)",
                   "superstep_us": [round(x, 1) for x in step_us]},
        "supersteps": steps, "syncs_done": st["syncs_done"], "syncs_skipped": st["syncs_skipped"],
        "sync_pairs": st["sync_pairs"],
        "roofline": {"bound": "hbm", "achieved": bytes_step / (k_us * 1e-6) / 1e9, "peak": peaks["hbm_gbs"],
                     "unit": "GB/s", "frac": bytes_step / (k_us * 1e-6) / 1e9 / peaks["hbm_gbs"], "traffic": None,
                     "peak_source": peaks["source"], "kernel": "k_lp_slices, row and hub kernels (+ sync)",
                     "avg_superstep_us": k_us, "algorithmic_bytes_per_superstep": bytes_step},
        "clocks": clk.summary(),
    }
    print(json.dumps(line), flush=True)
    ctx.close()


def _pct(xs, q):
    return float(np.percentile(np.asarray(xs, dtype=np.float64), q)) if len(xs) else None


def serve_cpu_baseline(stream, graphs_host, budget_s=20.0):
    """The oracle answering the served stream in order on this host, one query
    at a time (single-threaded fp64 C), until about budget_s seconds pass."""
    import oracle
    t0 = time.perf_counter()
    done = 0
    for i in range(len(stream["t"])):
        g, kind = int(stream["graph"][i]), int(stream["kind"][i])
        n, src, dst, w, elig = graphs_host[g]
        s = int(elig[stream["pick"][i]])
        if kind == 0:
            oracle.sssp(n, src, dst, w, s)
        else:
            oracle.ppr(n, src, dst, s, synth.SERVE_DAMPING, synth.SERVE_ITERS)
        done += 1
        if time.perf_counter() - t0 > budget_s:
            break
    dt = time.perf_counter() - t0
    return {"value": done / dt, "unit": "queries/s", "cores": 1, "kind": "oracle",
            "sample": f"the first {done} queries of the served stream, in order, one at a time"}


def run_serve(args):
    """Serving: an open-loop Poisson stream of SSSP and personalized-PageRank
    queries over four resident R-MAT graphs (scales 18/20/22/24), answered by
    the continuous-batching server; latency = scheduled arrival -> result in
    pinned host memory. Beside it, the same queries answered one at a time by
    the single-query engine, and by the server with all of them queued at once."""
    import threading
    import torch
    from paper_2203_13005_gb300 import gxp
    rate, dur = args.serve_rate, args.serve_seconds
    ctx = gxp.Context(0)
    srv = gxp.Server(ctx)
    engines, elig, host = [], [], []
    t_load = time.perf_counter()
    scales = [int(x) for x in args.serve_scales.split(",")]
    served = [wl for wl in synth.SERVE_GRAPHS if wl.scale in scales]
    for wl in served:
        src, dst, w = wl.edges()
        n = wl.n_vertices
        srv.add_graph(n, src, dst, w)
        e = gxp.Context(0)
        e.create_graph(n, 1)
        e.load_coo(src, dst, w)
        engines.append(e)
        el = np.flatnonzero(np.bincount(src, minlength=n) > 0).astype(np.uint32)
        elig.append(el)
        host.append((n, src, dst, w, el) if wl.scale <= 20 and not args.no_cpu_baseline else None)
        del src, dst, w
    load_s = time.perf_counter() - t_load
    srv.start(priorities=args.serve_priorities)
    stream = synth.serve_stream(rate, dur, [len(e) for e in elig], synth.SERVE_SEED)
    N = len(stream["t"])
    srcs = np.array([elig[g][p] for g, p in zip(stream["graph"], stream["pick"])], dtype=np.uint32)
    nmax = max(wl.n_vertices for wl in served)
    buf = torch.empty(nmax, dtype=torch.int32, pin_memory=True)

    def submit(i):
        return srv.submit(int(stream["graph"][i]), int(stream["kind"][i]), int(srcs[i]),
                          synth.SERVE_DAMPING, synth.SERVE_ITERS)

    # warm-up: every (graph, kind) lane and every single-query engine once
    for _ in range(args.warmup):
        for g in range(len(engines)):
            for kind in (gxp.GXP_QUERY_SSSP, gxp.GXP_QUERY_PPR):
                srv.poll(srv.submit(g, kind, int(elig[g][0]), synth.SERVE_DAMPING, synth.SERVE_ITERS), buf)
    for g, e in enumerate(engines):
        e.run(gxp.GXP_ALGO_SSSP, int(elig[g][0]))
        e.run(gxp.GXP_ALGO_PPR, int(elig[g][0]), synth.SERVE_DAMPING, synth.SERVE_ITERS)

    def replay(rate_q, dur_q):
        """Open-loop replay of a Poisson stream at rate_q for dur_q seconds:
        latency = scheduled arrival -> result in pinned host memory."""
        st = synth.serve_stream(rate_q, dur_q, [len(e) for e in elig], synth.SERVE_SEED)
        n_q = len(st["t"])
        srcs_q = np.array([elig[g][p] for g, p in zip(st["graph"], st["pick"])], dtype=np.uint32)
        lock = threading.Lock()
        qidx = {}
        lat = np.full(n_q, np.nan)
        info = [None] * n_q
        finish = [0.0]
        t_base = [0.0]
        rep0 = srv.report()

        def collector():
            got = 0
            while got < n_q:
                q = srv.next_done(1000)
                if q == 0:
                    if time.perf_counter() - t_base[0] > dur_q + args.serve_drain:
                        break
                    continue
                with lock:
                    i = qidx.get(q)
                while i is None:   # submit() returned but the id is not recorded yet
                    time.sleep(1e-5)
                    with lock:
                        i = qidx.get(q)
                info[i] = srv.info(q)
                srv.poll(q, buf)
                t = time.perf_counter()
                lat[i] = t - (t_base[0] + st["t"][i])
                finish[0] = t
                got += 1

        col = threading.Thread(target=collector)
        with ClockSampler(0) as clk:
            t_base[0] = time.perf_counter() + 0.05
            col.start()
            for i in range(n_q):
                target = t_base[0] + st["t"][i]
                while True:
                    d = target - time.perf_counter()
                    if d <= 0:
                        break
                    time.sleep(d - 2e-4 if d > 5e-4 else 0)
                q = srv.submit(int(st["graph"][i]), int(st["kind"][i]), int(srcs_q[i]),
                               synth.SERVE_DAMPING, synth.SERVE_ITERS)
                with lock:
                    qidx[q] = i
            col.join()
        # whatever the drain limit left behind is collected before the next phase
        while True:
            q = srv.next_done(200)
            if q == 0:
                r = srv.report()
                if r["queued"] + r["running"] == 0:
                    break
                continue
            srv.poll(q, buf)
        rep = srv.report()
        done = ~np.isnan(lat)
        lat_ms = lat[done] * 1e3
        span = finish[0] - t_base[0]
        by = {}
        for g, wl in enumerate(served):
            for kind, kn in ((0, "sssp"), (1, "ppr")):
                sel = done & (st["graph"] == g) & (st["kind"] == kind)
                by[f"{kn}_rmat{wl.scale}"] = {"n": int(sel.sum()), "p50_ms": _pct(lat[sel] * 1e3, 50),
                                              "p99_ms": _pct(lat[sel] * 1e3, 99)}
        qms = [x["queue_ms"] for x in info if x]
        rms = [x["run_ms"] for x in info if x]
        return {
            "offered_qps": rate_q, "duration_s": dur_q, "submitted": int(n_q), "completed": int(done.sum()),
            "achieved_qps": float(done.sum() / span) if span > 0 else 0.0, "span_s": span,
            "backlog_at_end": int(n_q - done.sum()),
            "latency": {"p50_ms": _pct(lat_ms, 50), "p90_ms": _pct(lat_ms, 90), "p99_ms": _pct(lat_ms, 99),
                        "max_ms": float(lat_ms.max()) if len(lat_ms) else None,
                        "queue_p50_ms": _pct(qms, 50), "queue_p99_ms": _pct(qms, 99),
                        "run_p50_ms": _pct(rms, 50), "run_p99_ms": _pct(rms, 99), "by_lane": by},
            "lane_supersteps": {"sssp": rep["sssp_supersteps"] - rep0["sssp_supersteps"],
                                "ppr": rep["ppr_supersteps"] - rep0["ppr_supersteps"]},
            "clocks": clk.summary(),
        }

    main = replay(rate, dur)
    second = replay(args.serve_rate2, dur) if args.serve_rate2 > 0 else None
    # lower offered rates, shorter windows: the highest rate whose p99 stays under 1 s
    sweep = []
    for r in [float(x) for x in args.serve_sweep.split(",") if x.strip()]:
        res = replay(r, args.serve_sweep_seconds)
        sweep.append({"offered_qps": r, "achieved_qps": res["achieved_qps"], "completed": res["completed"],
                      "p50_ms": res["latency"]["p50_ms"], "p99_ms": res["latency"]["p99_ms"],
                      "backlog_at_end": res["backlog_at_end"]})
    tried = sweep + [{"offered_qps": rate, **main["latency"]}]
    if second is not None:
        tried.append({"offered_qps": args.serve_rate2, **second["latency"]})
    held = [x["offered_qps"] for x in tried if x.get("p99_ms") is not None and x["p99_ms"] < 1000.0]

    # closed loop on the first K queries: one at a time vs all queued at once
    K = min(N, args.serve_closed)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for i in range(K):
        e = engines[int(stream["graph"][i])]
        if stream["kind"][i] == 0:
            e.run(gxp.GXP_ALGO_SSSP, int(srcs[i]))
        else:
            e.run(gxp.GXP_ALGO_PPR, int(srcs[i]), synth.SERVE_DAMPING, synth.SERVE_ITERS)
        e.values(out=buf[:e.n_vertices].numpy().view(
            np.float32 if stream["kind"][i] else np.uint32))
    single_s = time.perf_counter() - t0
    t0 = time.perf_counter()
    mine = {submit(i) for i in range(K)}
    while mine:   # collect in order of completion
        q = srv.next_done(-1)
        srv.poll(q, buf)
        mine.discard(q)
    batched_s = time.perf_counter() - t0

    base = None
    if not args.no_cpu_baseline and any(h is not None for h in host):
        # bounded sample: the stream's queries on the scale-18 and scale-20 graphs
        keep = np.isin(stream["graph"], [i for i, h in enumerate(host) if h is not None])
        base = serve_cpu_baseline({k: v[keep] for k, v in stream.items()}, host)
        base["sample"] += " (its queries on the scale-18 and scale-20 graphs)"
    rep = srv.report()
    line = {
        "metric": "served-query p50/p99 latency", "value": main["achieved_qps"],
        "unit": "queries/s", "n_gpus": 1, "steps": 1, "warmup": args.warmup,
        "ms_per_step": main["span_s"] * 1e3, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "u32+f32", "data": "synthetic",
        "config": {"workload": "serve_rmat" + "_".join(str(wl.scale) for wl in served), "offered_qps": rate,
                   "duration_s": dur,
                   "mix": f"graph uniform over {len(served)}, SSSP/PPR 1:1, sources uniform over out-degree >= 1",
                   "ppr": {"damping": synth.SERVE_DAMPING, "iters": synth.SERVE_ITERS},
                   "max_slots": 64, "results_per_graph": 128, "priorities": bool(args.serve_priorities)},
        "latency": main["latency"],
        "submitted": main["submitted"], "completed": main["completed"], "backlog_at_end": main["backlog_at_end"],
        "lane_supersteps": main["lane_supersteps"],
        "at_lower_rate": second,
        "rate_sweep": sweep,
        "highest_rate_with_p99_under_1s": max(held) if held else None,
        "closed_loop": {"queries": int(K), "one_at_a_time_qps": K / single_s, "batched_qps": K / batched_s,
                        "speedup": single_s / batched_s},
        "server_device_bytes": rep["device_bytes"], "graph_load_s": load_s,
        "cpu_baseline": base, "clocks": main["clocks"],
    }
    print(json.dumps(line), flush=True)
    srv.stop()
    for e in engines:
        e.close()
    ctx.close()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="gxp", choices=["gxp", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--e2e-steps", type=int, default=5)
    ap.add_argument("--workload", default=WL.name,
                    choices=[WL.name, synth.SSSP_RMAT16.name, synth.SSSP_RMAT22.name, synth.MSSSP_RMAT24.name,
                             synth.CC_ER24_P8.name, "lp_er24_8parts", synth.SSSP_CLUSTERED24_P8.name,
                             "serve"],
                    help="extra workloads print their own line; the default is the headline")
    ap.add_argument("--cache-slots", type=int, default=0,
                    help="cc_er24_8parts: cached remote vertices per partition (0 = all, 4294967295 = none)")
    ap.add_argument("--cc-scale", type=int, default=24, help="cc_er24_8parts: log2 vertices (smaller for profiling)")
    ap.add_argument("--lp-parts", type=int, default=8, help="lp_er24_8parts: partitions (1 = one, renumbered)")
    ap.add_argument("--lp-scale", type=int, default=24, help="lp_er24_8parts: log2 vertices (smaller for profiling)")
    ap.add_argument("--lp-graph", default="er", choices=["er", "rmat"],
                    help="lp_er24_8parts: the ER graph, or symmetric R-MAT (power-law) at --lp-scale")
    ap.add_argument("--direction", default="auto", choices=sorted(DIRECTIONS),
                    help="sssp_rmat16: direction of the supersteps")
    ap.add_argument("--push-div", type=int, default=0, help="sssp_rmat16: auto pushes while frontier work x div <= E")
    ap.add_argument("--serve-rate", type=float, default=synth.SERVE_RATE, help="serve: offered queries/s")
    ap.add_argument("--serve-seconds", type=float, default=synth.SERVE_SECONDS, help="serve: arrival window")
    ap.add_argument("--serve-drain", type=float, default=60.0, help="serve: seconds allowed after the window")
    ap.add_argument("--serve-closed", type=int, default=1000, help="serve: queries of the closed-loop comparison")
    ap.add_argument("--serve-scales", default="18,20,22,24", help="serve: R-MAT scales of the served graphs")
    ap.add_argument("--serve-priorities", action="store_true", help="serve: smaller graphs' lanes first")
    ap.add_argument("--serve-sweep", default="", help="serve: further offered rates (comma-separated), "
                    "each replayed for --serve-sweep-seconds")
    ap.add_argument("--serve-sweep-seconds", type=float, default=8.0)
    ap.add_argument("--serve-rate2", type=float, default=800.0,
                    help="serve: a second open-loop run at this rate (0: none)")
    args = ap.parse_args()
    world, rank, local = dist_setup()
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")

    if args.impl == "reference":
        run_reference(args, world, rank)
        return
    if args.workload == synth.MSSSP_RMAT24.name:
        run_msssp(args)
        return
    if args.workload == synth.CC_ER24_P8.name:
        run_cc(args)
        return
    if args.workload == "lp_er24_8parts":
        return run_lp(args)
    if args.workload == synth.SSSP_CLUSTERED24_P8.name:
        return run_sync_skip(args)
    if args.workload in (synth.SSSP_RMAT16.name, synth.SSSP_RMAT22.name):
        run_sssp(args)
        return
    if args.workload == "serve":
        run_serve(args)
        return

    import torch
    from paper_2203_13005_gb300 import gxp

    pg = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
        pg = dist
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    src, dst, _ = WL.edges()
    n, m = WL.n_vertices, WL.n_edges
    base = base_all = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        base = cpu_baseline(src, dst, n, m)
        base_all = cpu_all_cores_pagerank(src, dst, n, m)

    stream = torch.cuda.Stream(device=dev)
    ctx = gxp.Context(local)
    ctx.set_stream(stream.cuda_stream)
    ctx.create_graph(n, 1)
    ctx.load_coo(src, dst)
    g, mm, a = gxp.TEMPLATES[gxp.GXP_ALGO_PAGERANK]
    lib, h = ctx.lib, ctx.h

    def one_step(evs=None):
        rc = lib.gxp_begin(h, gxp.GXP_ALGO_PAGERANK, 0, DAMPING)
        if rc:
            ctx._ck(rc)
        for i in range(ITERS):
            if evs is not None:
                evs[i][0].record(stream)
            rc = lib.gxp_superstep(h, gxp.GXP_ALGO_PAGERANK, g, mm, a, None)
            if rc:
                ctx._ck(rc)
            if evs is not None:
                evs[i][1].record(stream)

    with torch.cuda.stream(stream):
        for _ in range(args.warmup):
            one_step()
    torch.cuda.synchronize()
    # per-superstep kernel events of every timed step
    evs = [[(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
            for _ in range(ITERS)] for _ in range(args.steps)]
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    if pg:
        pg.barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        t_start.record(stream)
        for s in range(args.steps):
            one_step(evs[s])
        t_end.record(stream)
        torch.cuda.synchronize()
    if pg:
        pg.barrier()
    ms_total = t_start.elapsed_time(t_end)
    kernel_ms = [b.elapsed_time(e) for step in evs for (b, e) in step]
    if pg:
        t = torch.tensor([ms_total], device=dev)
        pg.all_reduce(t, op=pg.ReduceOp.MAX)
        ms_total = float(t.item())
    ms_per_step = ms_total / args.steps
    gteps = world * ITERS * m / (ms_per_step * 1e-3) / 1e9

    # end to end through the public API with host buffers: CSC from pinned host
    # memory -> load -> 20 supersteps -> ranks back into pinned host memory
    order = np.argsort(dst, kind="stable")
    col_ptr = torch.zeros(n + 1, dtype=torch.int64).pin_memory()
    np.cumsum(np.bincount(dst, minlength=n), out=col_ptr.numpy()[1:])
    csc_src = torch.from_numpy(np.ascontiguousarray(src[order]).view(np.int32)).pin_memory()
    ranks_h = torch.empty(n, dtype=torch.float32).pin_memory()
    del order
    e2e_times = []
    ctx2 = gxp.Context(local)
    ctx2.set_stream(stream.cuda_stream)
    for i in range(args.e2e_steps + 1):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ctx2.create_graph(n, 1)
        ctx2.load_partition(0, gxp.GXP_FMT_CSC, m, col_ptr, csc_src)
        ctx2.run(gxp.GXP_ALGO_PAGERANK, damping=DAMPING, max_steps=ITERS)
        ctx2.values(out=ranks_h)
        torch.cuda.synchronize()
        if i > 0:
            e2e_times.append(time.perf_counter() - t0)
    e2e_s = statistics.median(e2e_times)
    ctx2.close()

    if rank == 0:
        peaks = measured_peaks()
        bytes_launch = algorithmic_bytes(n, m)
        bytes_launch_old_rank = algorithmic_bytes_with_old_rank(n, m)
        avg_kernel_s = statistics.mean(kernel_ms) * 1e-3
        achieved = bytes_launch / avg_kernel_s / 1e9
        traffic = profiled_traffic()
        line = {
            "metric": METRIC, "value": gteps, "unit": "GTEPS", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": WL.name, "vertices": n, "edges": m, "supersteps_per_step": ITERS,
                       "damping": DAMPING, "parallelism": f"replicas{world}",
                       "l2": "inputs larger than L2: 256 MiB of edge indices per superstep vs 129 MB L2"},
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                         "frac": achieved / peaks["hbm_gbs"], "traffic": traffic,
                         "peak_source": peaks["source"], "algorithmic_bytes_per_launch": bytes_launch,
                         "frac_with_old_rank_read": bytes_launch_old_rank / avg_kernel_s / 1e9 / peaks["hbm_gbs"],
                         "kernel": "k_sweep<PR>", "avg_launch_us": avg_kernel_s * 1e6},
            "e2e": {"value": ITERS * m / e2e_s / 1e9, "unit": "GTEPS",
                    "h2d_bytes_per_step": 8 * (n + 1) + 4 * m, "d2h_bytes_per_step": 4 * n,
                    "ms_per_step": e2e_s * 1e3},
            # per step: the initial state, 20 supersteps
            "gpu_launches": args.steps * (ITERS + 1),
            "clocks": clk.summary(),
        }
        if base is not None:
            line["cpu_baseline"] = base
            line["cpu_baseline_all_cores"] = base_all
        print(json.dumps(line), flush=True)
    ctx.close()
    if pg:
        pg.destroy_process_group()


if __name__ == "__main__":
    main()
