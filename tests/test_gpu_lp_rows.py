"""Label propagation at the edges of its row classes: register-sorted rows
of every width, hash tables filled to their largest rows with all-distinct
labels (the passes of the largest shared-memory class, the global tables past
it), and supersteps in which few labels change and only the rows they reach
are recomputed. Bit for bit against the oracle after every superstep."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu

# every width of a slice, then the borders of the classes and of the passes
DEGREES = list(range(0, 34)) + [64, 255, 256, 257, 2047, 2048, 2049, 8192, 8193, 16_385, 65_536, 65_537]


def _steps(c, n, src, dst, cap):
    lab = c.values()
    for t in range(cap):
        ref, ch_ref = oracle.lp_step(n, src, dst, lab)
        assert c.superstep() == ch_ref, f"superstep {t + 1}"
        assert np.array_equal(c.values(), ref), f"superstep {t + 1}"
        lab = ref
        if ch_ref == 0:
            break


@pytest.mark.parametrize("repeat", [1, 7, 3000])   # vertices a source is drawn from, at most n / repeat
@pytest.mark.parametrize("parts,keep_ids", [(1, False), (1, True), (3, True)])
def test_rows_at_class_borders(parts, keep_ids, repeat):
    n = 100_000
    rng = np.random.default_rng(repeat)
    rows = rng.permutation(n)[: len(DEGREES)]
    dst = np.repeat(rows, DEGREES).astype(np.uint32)
    # distinct sources within a row (an arithmetic sequence modulo n), folded to repeat labels
    at = np.concatenate([np.arange(k) for k in DEGREES])
    src = ((at * 7919 + dst) % n // repeat).astype(np.uint32)
    back = rng.integers(0, n, 50_000, dtype=np.uint32)   # the rows' labels travel on
    src = np.concatenate([src, rng.choice(rows, 50_000).astype(np.uint32)])
    dst = np.concatenate([dst, back])
    with gxp.Context(0, keep_ids=keep_ids) as c:
        c.create_graph(n, parts)
        c.load_coo(src, dst)
        c.begin(gxp.GXP_ALGO_LP)
        _steps(c, n, src, dst, 6)


@pytest.mark.parametrize("mem_budget", [0, 6_000_000])   # the second has no room for the out-edge copy
def test_few_changes(mem_budget):
    """A settled graph disturbed at a few vertices: the change travels along
    a path while everything else stays, with rows of every class next to it."""
    n = 40_000
    rng = np.random.default_rng(3)
    a = np.arange(1, 30_000)
    src = np.concatenate([a - 1, a, np.repeat(a, 2)])          # a path whose vertices weigh their left neighbour twice
    dst = np.concatenate([a, a, np.repeat(a, 2)])
    src = np.concatenate([src, a - 1, a - 1, a - 1])
    dst = np.concatenate([dst, a, a, a])
    for v, k in ((30_001, 100), (30_002, 1000), (30_003, 5000)):   # larger rows fed by the path
        src = np.concatenate([src, rng.integers(0, 30_000, k)])
        dst = np.concatenate([dst, np.full(k, v)])
    src, dst = src.astype(np.uint32), dst.astype(np.uint32)
    with gxp.Context(0, mem_budget=mem_budget) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst)
        c.begin(gxp.GXP_ALGO_LP)
        lab = np.zeros(n, np.uint32)
        lab[0] = 5
        lab[20_000] = 9
        c.set_values(lab)
        _steps(c, n, src, dst, 12)
        v = c.values()
        v[100:140] = 77
        c.set_values(v)
        _steps(c, n, src, dst, 8)
        assert c.run(gxp.GXP_ALGO_LP, max_steps=15) == 15
        ref, steps, _ = oracle.lp(n, src, dst)
        assert np.array_equal(c.values(), ref)
