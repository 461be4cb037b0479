"""Captured graphs of batched SSSP across calls of one context: other block
sizes, the autotuner and other numbers of sources come in between, which may
replace the buffers a captured graph refers to. Bit for bit against the
oracle."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def graph():
    wl = synth.MSSSP_RMAT24.scaled(11)
    src, dst, w = wl.edges()
    n = wl.n_vertices
    sources = synth.sources_with_out_edges(n, src, 64, 5)
    refs = [oracle.sssp(n, src, dst, w, int(s))[0] for s in sources]
    return n, src, dst, w, sources, refs


# (block_edges, use_graph, streamed, sources) of successive calls; block_edges 0 = tuned
@pytest.mark.parametrize("calls", [
    [(9000, True, True, 64), (500, False, True, 64), (9000, True, True, 64)],     # more counters in between
    [(500, True, True, 64), (20_000, False, True, 64), (500, True, True, 64)],    # a larger ring in between
    [(9000, True, True, 64), (0, True, True, 64), (9000, True, True, 64)],        # the tuner in between
    [(9000, True, True, 64), (0, False, False, 64), (300, True, True, 64), (9000, True, True, 64)],
    [(2000, True, True, k) for k in (1, 4, 5, 8, 33, 64, 9, 32, 17, 16, 3, 64)],  # a graph per lane grouping, kept
])
def test_buffers_replaced_between_graph_runs(gpu, graph, calls):
    n, src, dst, w, sources, refs = graph
    with gxp.Context(0) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst, w)
        for block_edges, use_graph, streamed, k in calls:
            dist, _ = c.sssp_batch(sources[:k], streamed=streamed, block_edges=block_edges, use_graph=use_graph)
            for j in range(k):
                assert np.array_equal(dist[:, j], refs[j]), (block_edges, use_graph, j)
