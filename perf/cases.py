"""What this framework is used for, as cases that can be timed.

Each case goes through the public binding (``paper_2203_13005_gb300.gxp``) the
way a user's program does: a graph is made resident once, then runs, batches
or queries are answered over it, or a graph is loaded from host memory, run
and forgotten. Graphs are the repository's own kinds: R-MAT (a, b, c, d) =
(.57, .19, .19, .05) with edge factor 16, uniform (Erdős–Rényi) pairs stored
both ways, and planted communities laid on the partitions; weights are
U{1..100} (U{1..255} for batches and queries). They are generated on the GPU
from the seed alone.
"""
from __future__ import annotations

import ctypes
import math

import torch

from paper_2203_13005_gb300 import gxp

DAMPING = 0.85
ITERS = 20        # PageRank / personalized PageRank supersteps
LP_STEPS = 15     # the paper's cap on label propagation
RMAT = (0.57, 0.19, 0.19)
ALGOS = {"sssp": gxp.GXP_ALGO_SSSP, "cc": gxp.GXP_ALGO_CC, "pagerank": gxp.GXP_ALGO_PAGERANK,
         "ppr": gxp.GXP_ALGO_PPR, "lp": gxp.GXP_ALGO_LP}


def listed():
    return [
        # one superstep over a CSC in the caller's own device memory: the
        # smallest call there is, all latency
        {"name": "step_csc_rmat12", "kind": "step_csc", "algo": "sssp", "graph": "rmat",
         "n": 1 << 12, "m": 1 << 16, "w_hi": 100},
        # a shortest-path query on a small resident graph (R-MAT 16)
        {"name": "sssp_rmat16", "kind": "run", "algo": "sssp", "graph": "rmat",
         "n": 1 << 16, "m": 1 << 20, "w_hi": 100, "parts": 1},
        # the same on a large one: dense supersteps pull, sparse ones push
        {"name": "sssp_rmat22", "kind": "run", "algo": "sssp", "graph": "rmat",
         "n": 1 << 22, "m": 1 << 26, "w_hi": 100, "parts": 1},
        # the flagship: PageRank of a resident power-law graph
        {"name": "pagerank_rmat22", "kind": "run", "algo": "pagerank", "graph": "rmat",
         "n": 1 << 22, "m": 1 << 26, "w_hi": 0, "parts": 1},
        # a graph seen once: loaded from pinned host memory, ranked, the ranks
        # read back; its vertex count is no power of two
        {"name": "load_pagerank_1m", "kind": "load", "algo": "pagerank", "graph": "rmat",
         "n": 1_000_003, "m": 1 << 24, "w_hi": 0},
        # a personalized ranking on a mid-sized graph of odd size
        {"name": "ppr_rmat_200k", "kind": "run", "algo": "ppr", "graph": "rmat",
         "n": 200_003, "m": 3_200_001, "w_hi": 0, "parts": 1},
        # connected components of a uniform graph in eight partitions: lazy
        # upload and cached copies between them after every superstep (one
        # giant component and some small ones)
        {"name": "cc_er_3m_8parts", "kind": "run", "algo": "cc", "graph": "er",
         "n": 3_000_000, "m": 1 << 25, "w_hi": 0, "parts": 8},
        # shortest paths over eight communities, one superstep per call as an
        # upper system drives them; many supersteps, skipped exchanges
        {"name": "steps_clustered19_8parts", "kind": "steps", "algo": "sssp", "graph": "clustered",
         "n": 1 << 19, "m": 1 << 23, "w_hi": 100, "parts": 8},
        # label propagation (15 supersteps) on a social-like graph with hubs,
        # edges stored both ways
        {"name": "lp_rmat20", "kind": "run", "algo": "lp", "graph": "rmat_both",
         "n": 1 << 20, "m": 1 << 25, "w_hi": 0, "parts": 1},
        # and on a uniform graph in eight partitions
        {"name": "lp_er20_8parts", "kind": "run", "algo": "lp", "graph": "er",
         "n": 1 << 20, "m": 1 << 24, "w_hi": 0, "parts": 8},
        # 64 sources at once, edges resident
        {"name": "batch64_rmat20", "kind": "batch", "graph": "rmat",
         "n": 1 << 20, "m": 1 << 24, "w_hi": 255, "sources": 64, "streamed": False},
        # the query server under a burst: 32 queries of each kind on each of
        # three resident graphs
        {"name": "serve_burst", "kind": "serve", "graph": "rmat",
         "n": 1 << 19, "m": 1 << 23, "w_hi": 255, "queries": 32, "graphs": 3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step_csc", "run", "run", "run", "run", "load", "steps", "batch", "serve"])
    if kind == "step_csc":
        n = _log(rng, 1 << 10, 1 << 20)
        algo = rng.choice(["sssp", "cc"])
        return {"kind": kind, "algo": algo, "graph": "rmat", "n": n, "m": n * rng.randint(4, 24) + rng.randint(0, 7),
                "w_hi": 100 if algo == "sssp" else 0}
    if kind == "run":
        algo = rng.choice(["sssp", "cc", "pagerank", "ppr", "lp"])
        parts = 1 if algo in ("pagerank", "ppr") else rng.choice([1, 1, 2, 5, 8])
        if parts > 1:
            graph, n = "er", _log(rng, 1 << 14, 1 << 20)
        elif algo in ("cc", "lp"):
            graph, n = rng.choice(["rmat_both", "er"]), _log(rng, 1 << 14, 1 << 20)
        else:
            graph, n = "rmat", _log(rng, 1 << 13, 3 << 20)
        # uniform graphs of more than about 8 edges a vertex are one component
        m = n * (rng.randint(3, 8) if algo == "cc" and graph == "er" else rng.randint(6, 16))
        return {"kind": kind, "algo": algo, "graph": graph, "n": n, "m": m - m % 2,
                "w_hi": 100 if algo == "sssp" else 0, "parts": parts}
    if kind == "load":
        n = _log(rng, 1 << 14, 1 << 20)
        algo = rng.choice(["pagerank", "sssp"])
        return {"kind": kind, "algo": algo, "graph": "rmat", "n": n, "m": n * rng.randint(6, 16) + rng.randint(0, 7),
                "w_hi": 100 if algo == "sssp" else 0}
    if kind == "steps":
        n = _log(rng, 1 << 14, 1 << 19)
        return {"kind": kind, "algo": "sssp", "graph": rng.choice(["clustered", "er"]), "n": n,
                "m": 2 * (n * rng.randint(3, 8)), "w_hi": 100, "parts": rng.choice([2, 4, 8])}
    if kind == "batch":
        n = _log(rng, 1 << 14, 1 << 20)
        return {"kind": kind, "graph": "rmat", "n": n, "m": n * rng.randint(8, 16), "w_hi": 255,
                "sources": rng.choice([5, 16, 33, 64, 64]), "streamed": rng.choice([False, False, True])}
    n = _log(rng, 1 << 14, 1 << 19)
    return {"kind": "serve", "graph": "rmat", "n": n, "m": n * rng.randint(8, 16), "w_hi": 255,
            "queries": rng.choice([1, 7, 32]), "graphs": rng.choice([1, 2, 3])}


# ------------------------------------------------------------------ inputs

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _edges(case, n, m, g):
    """Directed edges (src, dst) as int32 tensors."""
    dev = g.device
    if case["graph"].startswith("rmat"):
        both = case["graph"] == "rmat_both"
        k = m // 2 if both else m
        a, b, c = RMAT
        bits = max(1, (n - 1).bit_length())
        src = torch.zeros(k, dtype=torch.int32, device=dev)
        dst = torch.zeros(k, dtype=torch.int32, device=dev)
        for _ in range(bits):
            r = torch.rand(k, generator=g, device=dev)
            s = r >= a + b
            d = ((r >= a) & (r < a + b)) | (r >= a + b + c)
            src.mul_(2).add_(s)
            dst.mul_(2).add_(d)
        if n != 1 << bits:   # keep the skew on any vertex count
            src = ((src.long() * n) >> bits).int()
            dst = ((dst.long() * n) >> bits).int()
        return (torch.cat([src, dst]), torch.cat([dst, src])) if both else (src, dst)
    k = m // 2
    u = torch.randint(0, n, (k,), generator=g, device=dev)
    if case["graph"] == "er":
        v = (u + torch.randint(1, n, (k,), generator=g, device=dev)) % n
    else:   # communities on the partitions, one pair in 100,000 crossing
        bounds = torch.tensor(_bounds(n, case["parts"]), device=dev)
        p = torch.searchsorted(bounds, u, right=True) - 1
        lo, size = bounds[p], bounds[p + 1] - bounds[p]
        r = torch.rand(k, generator=g, device=dev, dtype=torch.float64)
        v = lo + (r * size).long().clamp(max=n)
        v = torch.minimum(v, lo + size - 1)
        cross = torch.rand(k, generator=g, device=dev) < 1e-5
        v = torch.where(cross, torch.randint(0, n, (k,), generator=g, device=dev), v)
    u, v = u.int(), v.int()
    return torch.cat([u, v]), torch.cat([v, u])


def _bounds(n, parts):
    return [n * p // parts for p in range(parts + 1)]


def _graph(case, seed, n, m):
    """Destination-sorted in-edges: offsets (int64), sources and weights
    (int32, the bits of the binding's uint32), and the out-degrees."""
    g = torch.Generator(device=_device())
    g.manual_seed(seed)
    src, dst = _edges(case, n, m, g)
    order = torch.sort(dst, stable=True).indices
    col = torch.zeros(n + 1, dtype=torch.int64, device=src.device)
    torch.cumsum(torch.bincount(dst, minlength=n), 0, out=col[1:])
    out_deg = torch.bincount(src, minlength=n)
    src = src[order]
    w = None
    if case["w_hi"]:
        w = torch.randint(1, case["w_hi"] + 1, (src.numel(),), generator=g, device=src.device, dtype=torch.int32)
    return col, src, w, out_deg, g


def _sources(out_deg, k, g):
    """k vertices drawn among those with an out-edge."""
    eligible = torch.nonzero(out_deg).flatten()
    pick = torch.randint(0, eligible.numel(), (k,), generator=g, device=eligible.device)
    return [int(v) for v in eligible[pick].tolist()]


def _serve_sizes(case):
    """The served graphs: each a quarter of the one before."""
    return [(max(case["n"] >> (2 * i), 64), max(case["m"] >> (2 * i), 1024)) for i in range(case["graphs"])]


def _inputs(case, seed):
    """What is computed on: also all that exact() needs."""
    if case["kind"] == "serve":
        got = []
        for i, (n, m) in enumerate(_serve_sizes(case)):
            col, src, w, out_deg, g = _graph(case, seed * 8 + i, n, m)
            got.append((n, col, src, w, out_deg, _sources(out_deg, 2 * case["queries"], g)))
        return got
    col, src, w, out_deg, g = _graph(case, seed, case["n"], case["m"])
    return col, src, w, out_deg, _sources(out_deg, case.get("sources", 1), g), g


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        ctx = gxp.Context(0)
        srv = gxp.Server(ctx)
        st = {"kind": kind, "ctx": ctx, "srv": srv, "queries": case["queries"], "sources": [], "out": []}
        for n, col, src, w, _, sources in _inputs(case, seed):
            dst = torch.repeat_interleave(torch.arange(n, device=src.device, dtype=torch.int32), col.diff())
            torch.cuda.synchronize()
            srv.add_graph(n, src, dst, w)
            st["sources"].append(sources)
            st["out"].append({"sssp": torch.empty(case["queries"], n, dtype=torch.int32, device=src.device),
                              "ppr": torch.empty(case["queries"], n, dtype=torch.float32, device=src.device)})
        srv.start()
        return st
    col, src, w, _, sources, g = _inputs(case, seed)
    n, m = case["n"], src.numel()
    if kind == "step_csc":
        # values half way through a run: some vertices reached, some not
        cur = torch.randint(0, 1000, (n,), generator=g, device=src.device, dtype=torch.int32)
        if case["algo"] == "sssp":
            cur[torch.rand(n, generator=g, device=src.device) < 0.5] = -1
        return {"kind": kind, "algo": ALGOS[case["algo"]], "n": n, "m": m, "col": col.int(), "src": src, "w": w,
                "cur": cur, "next": torch.empty_like(cur), "lib": gxp.load()}
    ctx = gxp.Context(0)
    st = {"kind": kind, "ctx": ctx, "source": sources[0], "n": n, "m": m, "w": w}
    if kind == "load":
        pin = lambda t: None if t is None else t.cpu().pin_memory()  # noqa: E731
        st.update(algo=ALGOS[case["algo"]], col=pin(col), src=pin(src), w=pin(w),
                  out=torch.empty(n, dtype=torch.float32 if case["algo"] == "pagerank" else torch.int32).pin_memory())
        return st
    parts = case.get("parts", 1)
    bounds = _bounds(n, parts)
    torch.cuda.synchronize()   # the context works on a stream of its own
    ctx.create_graph(n, parts)
    cuts = col[torch.tensor(bounds, device=col.device)].tolist()
    for p in range(parts):
        lo, hi = cuts[p], cuts[p + 1]
        offsets = col[bounds[p]:bounds[p + 1] + 1] - lo
        torch.cuda.synchronize()
        ctx.load_partition(p, gxp.GXP_FMT_CSC, hi - lo, offsets, src[lo:hi], None if w is None else w[lo:hi])
    if kind == "batch":
        st.update(sources=sources, streamed=case["streamed"], block=-(-m // 8),
                  out=torch.empty(n, len(sources), dtype=torch.int32, device=src.device))
        return st
    floats = case["algo"] in ("pagerank", "ppr")
    limit = ITERS if floats else LP_STEPS if case["algo"] == "lp" else 1 << 30
    st.update(algo=ALGOS[case["algo"]], limit=limit,
              out=torch.empty(n, dtype=torch.float32 if floats else torch.int32, device=src.device))
    return st


def run(st):
    kind = st["kind"]
    if kind == "step_csc":
        changed = ctypes.c_uint64()
        ptr = lambda t: None if t is None else t.data_ptr()  # noqa: E731
        rc = st["lib"].gxp_superstep_min_noalloc(st["algo"], st["n"], st["m"], ptr(st["col"]), ptr(st["src"]),
                                                 ptr(st["w"]), ptr(st["cur"]), ptr(st["next"]),
                                                 ctypes.byref(changed), None)
        if rc:
            raise RuntimeError("superstep failed: %d" % rc)
        return {"next": st["next"], "changed": changed.value}
    if kind == "serve":
        srv, k, asked = st["srv"], st["queries"], []
        for i in range(k):   # a burst: every graph and kind in turn
            for g, sources in enumerate(st["sources"]):
                asked.append((srv.submit(g, gxp.GXP_QUERY_SSSP, sources[i]), st["out"][g]["sssp"][i]))
                asked.append((srv.submit(g, gxp.GXP_QUERY_PPR, sources[k + i], DAMPING, ITERS), st["out"][g]["ppr"][i]))
        for query, out in asked:
            srv.poll(query, out)
        return st["out"]
    ctx = st["ctx"]
    if kind == "batch":
        ctx.sssp_batch(st["sources"], out=st["out"], streamed=st["streamed"],
                       block_edges=st["block"] if st["streamed"] else 0)
        return st["out"]
    if kind == "steps":
        ctx.begin(st["algo"], st["source"])
        steps = 1
        while ctx.superstep():
            steps += 1
    elif kind == "load":
        ctx.create_graph(st["n"], 1)
        ctx.load_partition(0, gxp.GXP_FMT_CSC, st["m"], st["col"], st["src"], st["w"])
        steps = ctx.run(st["algo"], st["source"], DAMPING, ITERS if st["algo"] == gxp.GXP_ALGO_PAGERANK else 1 << 30)
    else:
        steps = ctx.run(st["algo"], st["source"], DAMPING, st["limit"])
    return {"values": ctx.values(out=st["out"]), "supersteps": steps}


# ------------------------------------------------- what a pass cannot do without

def work(case):
    kind = case["kind"]
    per_edge = 8 if case["w_hi"] else 4   # source id (and weight)
    if kind == "serve":
        per = sum(8 * m + 4 * (n + 1) + 8 * case["queries"] * n for n, m in _serve_sizes(case))
        return {"bytes": per, "flops": sum(2 * ITERS * case["queries"] * m for _, m in _serve_sizes(case))}
    n, m = case["n"], case["m"]
    if kind == "batch":
        return {"bytes": 8 * m + 4 * (n + 1) + 4 * case["sources"] * n, "flops": case["sources"] * m}
    if kind == "step_csc":
        return {"bytes": per_edge * m + 4 * (n + 1) + 8 * n, "flops": m}
    if case["algo"] in ("pagerank", "ppr"):
        # every superstep reads each edge's source and gathers its message, and
        # reads and writes the vertices' state
        sweep = 8 * m + 16 * n
        loaded = 4 * m + 8 * (n + 1) if kind == "load" else 0
        return {"bytes": loaded + ITERS * sweep + 4 * n, "flops": ITERS * 2 * m}
    if case["algo"] == "lp":
        return {"bytes": 8 * m + 12 * n, "flops": m}   # one sweep: supersteps depend on the graph
    return {"bytes": (per_edge + 4) * m + 12 * n, "flops": m}


# ------------------------------------------------------------ in 64 bits

def _messages(col, src, out_deg, n):
    """A^T D^-1 in 64 bits: row v holds 1 / outdeg(u) for each in-edge (u, v)."""
    values = (1.0 / out_deg.clamp(min=1).double())[src.long()]
    return torch.sparse_csr_tensor(col, src.long(), values, size=(n, n))


def _ppr(col, src, out_deg, n, sources):
    a = _messages(col, src, out_deg, n)
    k = len(sources)
    at = (torch.tensor(sources, device=src.device), torch.arange(k, device=src.device))
    r = torch.zeros(n, k, dtype=torch.float64, device=src.device)
    r[at] = 1.0
    dangling = (out_deg == 0).double()
    for _ in range(ITERS):
        back = (1.0 - DAMPING) + DAMPING * (dangling @ r)
        r = DAMPING * (a @ r)
        r[at] += back
    return r


def _pagerank(col, src, out_deg, n):
    a = _messages(col, src, out_deg, n)
    r = torch.full((n, 1), 1.0 / n, dtype=torch.float64, device=src.device)
    dangling = (out_deg == 0).double()
    for _ in range(ITERS):
        r = (1.0 - DAMPING) / n + DAMPING * (dangling @ r) / n + DAMPING * (a @ r)
    return r[:, 0]


def exact(case, seed):
    """The fp32 results (ranks) in 64 bits; whole numbers have no entry."""
    if case["kind"] == "serve":
        return [{"sssp": None, "ppr": _ppr(col, src, out_deg, n, sources[case["queries"]:]).T.contiguous()}
                for n, col, src, _, out_deg, sources in _inputs(case, seed)]
    if case.get("algo") not in ("pagerank", "ppr"):
        return None
    col, src, _, out_deg, sources, _ = _inputs(case, seed)
    if case["algo"] == "ppr":
        return {"values": _ppr(col, src, out_deg, case["n"], sources)[:, 0], "supersteps": None}
    r = _pagerank(col, src, out_deg, case["n"])
    return {"values": r.cpu() if case["kind"] == "load" else r, "supersteps": None}
