"""gxp_stats.edges_scanned of label propagation on one partition: every edge in
a superstep that recomputes every row, else the in-edges of the rows that a
change reaches (the changed vertices and their out-neighbours)."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("keep_ids", [False, True])
def test_edges_of_supersteps_that_recompute_some_rows(gpu, keep_ids):
    n = 40_000
    rng = np.random.default_rng(3)
    a = np.arange(1, 30_000)
    src = np.concatenate([a - 1, a - 1, a - 1, a, a])   # a path whose vertices weigh their left neighbour more
    dst = np.tile(a, 5)
    for v, k in ((30_001, 100), (30_002, 1000), (30_003, 5000), (30_004, 70_000)):   # rows of the other classes, fed by the path
        src = np.concatenate([src, rng.integers(0, 30_000, k)])
        dst = np.concatenate([dst, np.full(k, v)])
    src, dst = src.astype(np.uint32), dst.astype(np.uint32)
    m, indeg, outdeg = len(src), np.bincount(dst, minlength=n), np.bincount(src, minlength=n)
    with gxp.Context(0, keep_ids=keep_ids) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst)
        c.begin(gxp.GXP_ALGO_LP)
        lab = np.zeros(n, np.uint32)
        lab[0], lab[20_000] = 5, 9
        c.set_values(lab)
        seen, expect, some = 0, m, 0   # the first superstep recomputes every row
        for t in range(8):
            new, changed = oracle.lp_step(n, src, dst, lab)
            assert c.superstep() == changed
            assert np.array_equal(c.values(), new)
            total = c.stats()["edges_scanned"]
            assert total - seen == expect, t
            seen = total
            ch = np.flatnonzero(new != lab)
            lab = new
            if outdeg[ch].sum() * 8 <= m:
                rows = np.union1d(ch, dst[np.isin(src, ch)])
                expect, some = int(indeg[rows].sum()), some + 1
            else:
                expect = m
        assert some >= 4
        assert c.stats()["push_supersteps"] == 0
