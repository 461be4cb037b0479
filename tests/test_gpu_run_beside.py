"""gxp_run of one partition beside other work on the GPU: a kernel that holds an
SM for a while (a bounded sleep on another stream), and a query server that
answers a fixed number of queries. The runs finish with the oracle's results
and do not wait for the other work to end."""
import time

import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def graph():
    wl = synth.SSSP_RMAT16.scaled(17)   # enough work for a CTA on every SM
    src, dst, w = wl.edges()
    return wl.n_vertices, src, dst, w


def _refs(graph):
    n, src, dst, w = graph
    return {gxp.GXP_ALGO_SSSP: oracle.sssp(n, src, dst, w, 0), gxp.GXP_ALGO_CC: oracle.cc(n, src, dst),
            gxp.GXP_ALGO_PAGERANK: oracle.pagerank(n, src, dst, 0.85, 40)}


def _run(c, algo, ref):
    if algo == gxp.GXP_ALGO_PAGERANK:
        assert c.run(algo, max_steps=40) == 40   # two launches of up to 32 supersteps
        r = c.values().astype(np.float64)
        assert (np.abs(r - ref[0]) / ref[0]).max() <= 1e-4
        assert np.abs(r - ref[0]).sum() <= 1e-5
    else:
        assert c.run(algo, source=0) == ref[1]
        assert np.array_equal(c.values(), ref[0])


@pytest.mark.parametrize("algo", [gxp.GXP_ALGO_SSSP, gxp.GXP_ALGO_CC, gxp.GXP_ALGO_PAGERANK])
def test_beside_a_sleeping_kernel(gpu, graph, algo):
    import torch
    ref = _refs(graph)[algo]
    with gxp.Context(0) as c:
        c.create_graph(graph[0], 1)
        c.load_coo(*graph[1:])
        _run(c, algo, ref)
        assert c.stats()["persistent_launches"] >= 1
        torch.cuda._sleep(1000)   # loaded
        torch.cuda.synchronize()
        t = time.perf_counter()
        torch.cuda._sleep(20_000_000)
        torch.cuda.synchronize()
        rate = 20_000_000 / (time.perf_counter() - t)
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            torch.cuda._sleep(int(0.4 * rate))
        time.sleep(0.02)   # it is running
        _run(c, algo, ref)
        assert c.stats()["persistent_launches"] == 0
        assert not side.query()   # the run did not wait for it
        torch.cuda.synchronize()
        _run(c, algo, ref)
        assert c.stats()["persistent_launches"] >= 1


def test_beside_a_query_server(gpu, graph):
    n, src, dst, w = graph
    refs = _refs(graph)
    with gxp.Context(0) as sc, gxp.Context(0) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst, w)
        server = gxp.Server(sc)
        graphs = [server.add_graph(n, src, dst, w) for _ in range(2)]
        server.start(priorities=True)
        queries = [(server.submit(g, kind, v, iters=20), kind, g)
                   for v in range(100) for g in graphs for kind in (gxp.GXP_QUERY_SSSP, gxp.GXP_QUERY_PPR)]
        for _ in range(5):
            for algo, ref in refs.items():
                _run(c, algo, ref)
        for q, kind, g in queries:
            r = server.result(q, kind, g)
            assert r.shape == (n,)
        assert server.report()["completed"] == len(queries)
        server.stop()
