"""Label propagation on a weighted graph next to SSSP and CC on the same one:
its out-edge copy holds no weights, theirs does. Bit for bit against the
oracle."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("direction", [gxp.GXP_DIR_AUTO, gxp.GXP_DIR_PUSH])
@pytest.mark.parametrize("order", ["lp sssp lp", "sssp lp cc", "lp cc sssp lp sssp"])
def test_in_any_order(gpu, order, direction):
    n, m = 3000, 20_000
    rng = np.random.default_rng(5)
    src, dst = rng.integers(0, n, m).astype(np.uint32), rng.integers(0, n, m).astype(np.uint32)
    w = rng.integers(1, 100, m).astype(np.uint32)
    refs = {"lp": oracle.lp(n, src, dst), "sssp": oracle.sssp(n, src, dst, w, 9), "cc": oracle.cc(n, src, dst)}
    algos = {"lp": gxp.GXP_ALGO_LP, "sssp": gxp.GXP_ALGO_SSSP, "cc": gxp.GXP_ALGO_CC}
    with gxp.Context(0, direction=direction) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst, w)
        for name in order.split():
            steps = c.run(algos[name], source=9, max_steps=15 if name == "lp" else 1 << 30)
            assert steps == refs[name][1], name
            assert np.array_equal(c.values(), refs[name][0]), name


def test_no_room_taken_for_weights(gpu):
    """What label propagation adds to the device memory of a loaded graph does
    not depend on the weights."""
    n, m = 3000, 100_000
    rng = np.random.default_rng(6)
    src, dst = rng.integers(0, n, m).astype(np.uint32), rng.integers(0, n, m).astype(np.uint32)
    added = []
    for w in (None, rng.integers(1, 100, m).astype(np.uint32)):
        with gxp.Context(0) as c:
            c.create_graph(n, 1)
            c.load_coo(src, dst, w)
            c.run(gxp.GXP_ALGO_PAGERANK, max_steps=1)   # the layout, which holds the weights
            before = c.stats()["device_bytes"]
            c.run(gxp.GXP_ALGO_LP, max_steps=15)
            added.append(c.stats()["device_bytes"] - before)
    assert added[0] == added[1]
