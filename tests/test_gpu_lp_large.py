"""Label propagation on partitions whose labels and copies do not fit L2: a warp
per slice instead of a striding grid. Bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,parts", [(12_000_000, 8), (45_000_037, 1)])   # 180 MB of labels and copies, each
def test_copies_past_l2(n, parts):
    m = 48_000_000
    rng = np.random.default_rng(n)
    src = rng.integers(0, n, m, dtype=np.uint32)
    dst = rng.integers(0, n, m, dtype=np.uint32)
    ref, _, _ = oracle.lp(n, src, dst, 2)
    with gxp.Context(0) as c:
        c.create_graph(n, parts)
        c.load_coo(src, dst)
        c.run(gxp.GXP_ALGO_LP, max_steps=2)
        assert np.array_equal(c.values(), ref)
