"""Label propagation over rows of up to 65,536 in-edges whose labels crowd under
the hashes of the row's shared-memory table: under the one that deals labels to
passes (the first try would need hundreds of thousands of them), under the one
that gives a label its first slot, or under both. Against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu

PASS_HASH, SLOT_HASH = 0x85EBCA6B, 0x9E3779B1


def _labels(kind, k):
    i = np.arange(1, k + 1, dtype=np.uint64)
    if kind == "pass":      # consecutive under the first
        i = i * pow(PASS_HASH, -1, 1 << 32)
    elif kind == "slot":    # consecutive under the second: one first slot for up to 2^18
        i = i * pow(SLOT_HASH, -1, 1 << 32)
    elif kind == "both":    # half and half
        i = np.where(i % 2 == 0, i * pow(PASS_HASH, -1, 1 << 32), i * pow(SLOT_HASH, -1, 1 << 32))
    return (i & 0xFFFFFFFF).astype(np.uint32)


def test_the_crowd_is_one():
    # (no GPU needed, but the sets only matter for the kernel) passes the first
    # hash alone would need until no pass holds more labels than 16,384 slots
    h = _labels("pass", 60_000).astype(np.uint64) * PASS_HASH & 0xFFFFFFFF
    passes = 8
    while np.bincount((h * passes >> np.uint64(32)).astype(np.int64)).max() > 16_384:
        passes *= 2
    assert passes == 262_144
    s = _labels("slot", 16_000).astype(np.uint64) * SLOT_HASH & 0xFFFFFFFF
    assert len(np.unique(s >> np.uint64(32 - 14))) == 1


@pytest.mark.parametrize("parts", [1, 2])
@pytest.mark.parametrize("kind", ["pass", "slot", "both", "none"])
def test_rows_of_crowded_labels(gpu, kind, parts):
    n = 70_000
    rng = np.random.default_rng(7)
    degrees = [2049, 4097, 8192, 8193, 16_384, 16_385, 60_000, 65_536]
    rows = n - 1 - np.arange(len(degrees))
    dst = np.repeat(rows, degrees).astype(np.uint32)
    src = np.concatenate([rng.permutation(66_000)[:d] for d in degrees]).astype(np.uint32)
    lab = np.empty(n, np.uint32)
    lab[:66_000] = _labels(kind, 66_000)
    lab[66_000:] = np.arange(66_000, n)
    with gxp.Context(0) as c:
        c.create_graph(n, parts)
        c.load_coo(src, dst)
        c.begin(gxp.GXP_ALGO_LP)
        for repeats in (0, 3):   # all labels distinct, then three vertices in a hundred share one
            x = lab.copy()
            if repeats:
                x[rng.integers(0, 66_000, 2000)] = x[5]
            c.set_values(x)
            ref, changed = oracle.lp_step(n, src, dst, x)
            assert c.superstep() == changed
            assert np.array_equal(c.values(), ref)
