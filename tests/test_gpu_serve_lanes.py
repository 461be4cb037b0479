"""Served personalized PageRank on graphs of different sizes: small ones widen
the lane groups and keep more rows in flight, large ones take both kernels as
the number of queries grows, and a few queries deal their units over the CTAs.
A query's result has the same bits alone and among others."""
import numpy as np
import pytest

from paper_2203_13005_gb300 import gxp, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 4_000, 20_000, 39_000, 100_000, 160_000])   # 16 .. 1 lanes a row alone
def test_bits_by_graph_size_and_queries(n):
    rng = np.random.default_rng(n)
    m = 6 * n
    src = (n * rng.random(m) ** 2).astype(np.uint32)
    dst = (n * rng.random(m) ** 3).astype(np.uint32)   # rows of up to many units
    sources = [int(s) for s in synth.sources_with_out_edges(n, src, min(64, n - 2), 9)]
    with gxp.Context(0) as ctx:
        srv = gxp.Server(ctx)
        g = srv.add_graph(n, src, dst, np.ones(m, np.uint32))
        first = {}
        for slots in (1, 2, 4, 5, 16, 64):
            srv.start(max_slots=slots, results_per_graph=128)
            ids = [(s, srv.submit(g, gxp.GXP_QUERY_PPR, s)) for s in sources[: 2 if slots == 1 else slots]]
            for s, q in ids:
                r = srv.result(q, gxp.GXP_QUERY_PPR, g)
                assert abs(float(r.astype(np.float64).sum()) - 1.0) < 1e-3
                assert np.array_equal(first.setdefault(s, r), r), (slots, s)
            srv.stop()
