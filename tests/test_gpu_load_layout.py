"""Loading a one-partition CSC: the sources arrive, are checked and counted in
chunks of at least 2^21 edges, and the renumbered rows are written 2,048 edges
at a time. Edge counts at the borders of both, rows that span many of them, and
a row per edge; weighted and not; a bad id in the last chunk is refused. Against
the oracle: SSSP bit for bit, PageRank within the fp32 bars of the other
superstep tests (relative 1e-4, L1 1e-5)."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu


def _csc(kind, m, seed):
    rng = np.random.default_rng(seed)
    n = {"path": m + 1, "star": 700, "mixed": max(m // 9, 3)}[kind]
    if kind == "path":      # one in-edge a row
        dst = 1 + rng.permutation(m)
    elif kind == "star":    # nearly all edges in one row
        dst = np.where(rng.random(m) < 0.9, 5, rng.integers(0, n, m))
    else:
        dst = (n * rng.random(m) ** 2).astype(np.int64)
    dst = np.sort(dst).astype(np.uint32)
    src = rng.integers(0, n, m).astype(np.uint32)
    w = rng.integers(1, 101, m).astype(np.uint32)
    col = np.concatenate([[0], np.cumsum(np.bincount(dst, minlength=n))]).astype(np.uint64)
    return n, col, src, dst, w


@pytest.mark.parametrize("keep_ids", [False, True])
@pytest.mark.parametrize("kind", ["path", "star", "mixed"])
@pytest.mark.parametrize("m", [1, 2047, 2048, 2049, (1 << 21) - 1, 1 << 21, (1 << 21) + 5])
def test_edges_at_chunk_borders(kind, m, keep_ids):
    n, col, src, dst, w = _csc(kind, m, m)
    source = int(src[0])
    d_ref, steps, _ = oracle.sssp(n, src, dst, w, source)
    r_ref, _, _ = oracle.pagerank(n, src, dst, 0.85, 4)
    with gxp.Context(0, keep_ids=keep_ids) as c:
        c.create_graph(n, 1)
        c.load_partition(0, gxp.GXP_FMT_CSC, m, col, src, w)
        assert c.run(gxp.GXP_ALGO_SSSP, source) == steps
        assert np.array_equal(c.values(), d_ref)
        c.load_partition(0, gxp.GXP_FMT_CSC, m, col, src, None)   # a new graph in the same context
        c.run(gxp.GXP_ALGO_PAGERANK, max_steps=4)
        r = c.values().astype(np.float64)
        nz = r_ref > 0
        assert np.all(r[~nz] == 0)
        assert (np.abs(r - r_ref)[nz] / r_ref[nz]).max() <= 1e-4
        assert np.abs(r - r_ref).sum() <= 1e-5


def test_bad_source_in_the_last_chunk():
    m = (1 << 21) + 5
    n, col, src, dst, w = _csc("mixed", m, 3)
    d_ref, _, _ = oracle.sssp(n, src, dst, w, 0)
    bad = src.copy()
    bad[-1] = n
    with gxp.Context(0) as c:
        c.create_graph(n, 1)
        with pytest.raises(gxp.GxpError):
            c.load_partition(0, gxp.GXP_FMT_CSC, m, col, bad, w)
        c.load_partition(0, gxp.GXP_FMT_CSC, m, col, src, w)
        c.run(gxp.GXP_ALGO_SSSP, 0)
        assert np.array_equal(c.values(), d_ref)
