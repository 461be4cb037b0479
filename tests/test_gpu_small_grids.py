"""Runs of one partition on graphs around the sizes at which the superstep
kernel starts to fill its CTAs (32 work items, a slice of 32 rows each, a CTA) and
the chip (152 of them), one graph after the other in the same context: bit for
bit against the oracle, ranks within 1e-4."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu

ITEMS = [1, 2, 31, 32, 33, 63, 64, 65, 151, 153, 32 * 151, 32 * 152 - 1, 32 * 152, 32 * 152 + 1]


@pytest.mark.parametrize("direction", [gxp.GXP_DIR_AUTO, gxp.GXP_DIR_PULL])
@pytest.mark.parametrize("timeout_ns", [0, 1_000_000])   # the second: a launch per superstep
def test_items_at_the_borders(gpu, direction, timeout_ns):
    with gxp.Context(0, direction=direction, timeout_ns=timeout_ns) as c:
        for items in ITEMS:
            n = 32 * items
            rng = np.random.default_rng(items)
            # one or two in-edges a row, a few chains among them
            dst = np.concatenate([np.arange(n), rng.integers(0, n, n // 2)]).astype(np.uint32)
            src = np.concatenate([np.maximum(np.arange(n) - 1, 0), rng.integers(0, n, n // 2)]).astype(np.uint32)
            w = rng.integers(1, 100, len(dst)).astype(np.uint32)
            c.create_graph(n, 1)
            c.load_coo(src, dst, w)
            d, steps, _ = oracle.sssp(n, src, dst, w, n // 2)
            assert c.run(gxp.GXP_ALGO_SSSP, source=n // 2) == steps, items
            assert np.array_equal(c.values(), d), items
            lab, steps, _ = oracle.cc(n, src, dst)
            assert c.run(gxp.GXP_ALGO_CC) == steps, items
            assert np.array_equal(c.values(), lab), items
            c.run(gxp.GXP_ALGO_PAGERANK, max_steps=35)
            r, ref = c.values().astype(np.float64), oracle.pagerank(n, src, dst, 0.85, 35)[0]
            assert (np.abs(r - ref) / ref).max() <= 1e-4, items


@pytest.mark.parametrize("direction", [gxp.GXP_DIR_AUTO, gxp.GXP_DIR_PULL, gxp.GXP_DIR_PUSH])
@pytest.mark.parametrize("algo", [gxp.GXP_ALGO_SSSP, gxp.GXP_ALGO_CC])
def test_superstep_after_a_run(gpu, algo, direction):
    """A run of launches of their own ends in supersteps enqueued past the fixed
    point, which return at once; supersteps driven by the caller go on from there."""
    n = 3000
    rng = np.random.default_rng(8)
    src, dst = rng.integers(0, n, 9000).astype(np.uint32), rng.integers(0, n, 9000).astype(np.uint32)
    w = rng.integers(1, 100, 9000).astype(np.uint32)
    sssp = algo == gxp.GXP_ALGO_SSSP
    ref, steps, _ = oracle.sssp(n, src, dst, w, 4) if sssp else oracle.cc(n, src, dst)
    step = (lambda x: oracle.sssp_step(n, src, dst, w, x)) if sssp else (lambda x: oracle.cc_step(n, src, dst, x))
    with gxp.Context(0, timeout_ns=1000, direction=direction) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst, w)
        for _ in range(2):
            assert c.run(algo, source=4) == steps
            assert c.superstep() == 0
            assert np.array_equal(c.values(), ref)
            x = ref.copy()
            x[rng.integers(0, n, 5)] = 0
            c.set_values(x)
            for _ in range(6):
                x, changed = step(x)
                assert c.superstep() == changed
                assert np.array_equal(c.values(), x)


@pytest.mark.parametrize("timeout_ns,persistent", [(0, True), (500_000_000, True), (100_000_000, True), (99_999_999, False)])
def test_timeout_that_allows_barriers(gpu, timeout_ns, persistent):
    n = 1000
    src, dst = np.arange(n - 1, dtype=np.uint32), np.arange(1, n, dtype=np.uint32)
    with gxp.Context(0, timeout_ns=timeout_ns) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst)
        c.run(gxp.GXP_ALGO_PAGERANK, max_steps=5)
        assert (c.stats()["persistent_launches"] > 0) == persistent
