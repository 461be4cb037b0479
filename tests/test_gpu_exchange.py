"""The exchange after a run: gxp_run writes the global data queue only after
its last superstep, which is the one gxp_sync returns; a run cut short by
max_steps, one that settles, and supersteps driven one by one all leave the
oracle's uploads and skip flags, whatever the direction."""
import numpy as np
import pytest

import oracle
from oracle import sync as osync
from paper_2203_13005_gb300 import gxp, synth

pytestmark = pytest.mark.gpu


def _check(c, parts, uploads, skipped):
    for p in range(parts):
        ids, vals, sk = c.sync(p)
        assert sk == skipped
        assert np.array_equal(ids, uploads[p][0]) and np.array_equal(vals, uploads[p][1])


@pytest.mark.parametrize("parts", [2, 5])
@pytest.mark.parametrize("direction", [gxp.GXP_DIR_AUTO, gxp.GXP_DIR_PULL, gxp.GXP_DIR_PUSH])
def test_queue_after_runs(direction, parts):
    n = 6001   # partitions that start inside a bitmap word
    src, dst = synth.erdos_renyi(n, 9000, 17)
    bounds = [n * p // parts for p in range(parts + 1)]
    _, _, trace = osync.min_label_sync_trace(n, src, dst, bounds, "cc")
    _, steps_ref, _ = oracle.cc(n, src, dst)
    with gxp.Context(0, direction=direction) as c:
        c.create_graph(n, parts)
        c.load_coo(src, dst)
        for k in (1, 2, 5, steps_ref - 1):
            assert c.run(gxp.GXP_ALGO_CC, max_steps=k) == k
            _check(c, parts, *trace[k - 1])
        assert c.run(gxp.GXP_ALGO_CC) == steps_ref
        _check(c, parts, *trace[steps_ref - 1])
        c.run(gxp.GXP_ALGO_CC, max_steps=3)
        c.superstep()   # a superstep after a run goes on from its state
        _check(c, parts, *trace[3])
        assert c.stats()["sync_pairs"] == sum(len(ids) for uploads, _ in trace[:4] for ids, _ in uploads)
