"""Loading a graph whose edges leave one vertex: out-degrees (PageRank's
messages divide by them) are exact, and counting them does not depend on the
vertex's id."""
import time

import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu

N, M = 1 << 18, 1 << 23


def _star(hub):
    dst = np.sort(np.random.default_rng(1).integers(0, N, M)).astype(np.uint32)
    col = np.concatenate([[0], np.cumsum(np.bincount(dst, minlength=N))]).astype(np.uint64)
    return np.full(M, hub, np.uint32), dst, col


def test_hub_above_the_counters_in_shared_memory(gpu):
    # the time of a load, the shortest of several: 21 times as long when every
    # edge of a high id took its own atomic, 1.2 times now
    best = {}
    for hub in (5, N - 7):
        src, dst, col = _star(hub)
        with gxp.Context(0) as c:
            c.create_graph(N, 1)
            took = []
            for _ in range(5):
                t = time.perf_counter()
                c.load_partition(0, gxp.GXP_FMT_CSC, M, col, src)
                took.append(time.perf_counter() - t)
            best[hub] = min(took)
            c.run(gxp.GXP_ALGO_PAGERANK, max_steps=2)
            r = c.values().astype(np.float64)
        ref, _, _ = oracle.pagerank(N, src, dst, 0.85, 2)
        assert (np.abs(r - ref) / ref).max() <= 1e-4
    assert best[N - 7] < 3 * best[5]
