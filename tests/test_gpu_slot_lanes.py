"""Batched and served queries with every number of lanes a row of slots can
take (1, 2, 4, 8 or 16 lanes of four slots): batches of 1..64 sources with
small and saturating weights, resident and streamed, and served personalized
PageRank whose results have the same bits however many queries run beside
them."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp, synth

pytestmark = pytest.mark.gpu


def _graph(n, m, w_hi, seed):
    rng = np.random.default_rng(seed)
    src = (n * rng.random(m) ** 2).astype(np.uint32)   # rows and out-degrees of many sizes, one over 256 in-edges
    dst = (n * rng.random(m) ** 3).astype(np.uint32)
    w = rng.integers(0, w_hi + 1, m, dtype=np.uint64).astype(np.uint32)
    return src, dst, w


def _distances(n, src, dst, w, s):
    """Bellman-Ford in 64 bits; distances past 32 bits read 0xFFFFFFFE, as the
    superstep's sums saturate (the oracle does not: it covers distances below
    that)."""
    d = np.full(n, 1 << 62, np.int64)
    d[s] = 0
    for _ in range(n):
        nd = d.copy()
        np.minimum.at(nd, dst, d[src] + w.astype(np.int64))
        if np.array_equal(nd, d):
            break
        d = nd
    return np.where(d >= 1 << 61, 0xFFFFFFFF, np.minimum(d, 0xFFFFFFFE)).astype(np.uint32)


@pytest.mark.parametrize("k", [1, 4, 5, 8, 9, 16, 17, 32, 33, 64])
@pytest.mark.parametrize("w_hi", [255, 0xFFFFFFFF])   # the second saturates and does not pack
def test_batch_source_counts(k, w_hi):
    n = 3000
    src, dst, w = _graph(n, 40_000, w_hi, k)
    sources = synth.sources_with_out_edges(n, src, k, 7)
    with gxp.Context(0) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst, w)
        a, _ = c.sssp_batch(sources)
        b, _ = c.sssp_batch(sources, streamed=True, block_edges=7000)
        g, _ = c.sssp_batch(sources[: (k + 1) // 2], use_graph=True, streamed=True, block_edges=7000)
    for j, s in enumerate(sources):
        ref = _distances(n, src, dst, w, int(s))
        assert np.array_equal(a[:, j], ref) and np.array_equal(b[:, j], ref), j
        if j < g.shape[1]:
            assert np.array_equal(g[:, j], ref), j


def test_served_pagerank_bits_by_queries_in_flight():
    n = 3000
    src, dst, w = _graph(n, 40_000, 255, 3)
    sources = [int(s) for s in synth.sources_with_out_edges(n, src, 64, 9)]
    with gxp.Context(0) as ctx:
        srv = gxp.Server(ctx)
        g = srv.add_graph(n, src, dst, w)
        alone = {}
        for slots in (1, 3, 8, 16, 32, 64):   # at most that many queries share a superstep
            srv.start(max_slots=slots, results_per_graph=128)
            ids = [(s, srv.submit(g, gxp.GXP_QUERY_PPR, s), srv.submit(g, gxp.GXP_QUERY_SSSP, s))
                   for s in sources[:max(4, slots)]]
            for s, p, q in ids:
                r = srv.result(p, gxp.GXP_QUERY_PPR, g)
                d = srv.result(q, gxp.GXP_QUERY_SSSP, g)
                if s in alone:
                    assert np.array_equal(alone[s], r), (slots, s)
                else:
                    alone[s] = r
                    assert np.array_equal(d, oracle.sssp(n, src, dst, w, s)[0])
            srv.stop()
