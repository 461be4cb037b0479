"""A graph loaded over another one in the same context: whatever was kept of
the first (host copies for the batched path among it) is forgotten. Bit for bit
against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu

N = 3001
SOURCES = np.array([0, 7, 1500], np.uint32)


def _edges(seed, m):
    rng = np.random.default_rng(seed)
    dst = np.sort(rng.integers(0, N, m)).astype(np.uint32)
    src = rng.integers(0, N, m).astype(np.uint32)
    w = rng.integers(1, 50, m).astype(np.uint32)
    return src, dst, w


def _load(c, fmt, src, dst, w):
    if fmt == gxp.GXP_FMT_COO:
        c.load_partition(0, fmt, len(src), src, dst, w)
    else:
        col = np.concatenate([[0], np.cumsum(np.bincount(dst, minlength=N))]).astype(np.uint64)
        c.load_partition(0, fmt, len(src), col, src, w)


def _check_batch(c, g, streamed):
    dist, _ = c.sssp_batch(SOURCES, streamed=streamed, block_edges=2000 if streamed else 0)
    for k, s in enumerate(SOURCES):
        ref, _, _ = oracle.sssp(N, *g, int(s))
        assert np.array_equal(dist[:, k], ref), f"source {s}"


@pytest.mark.parametrize("streamed", [False, True])
@pytest.mark.parametrize("first", [gxp.GXP_FMT_COO, gxp.GXP_FMT_CSC])
def test_batch_after_a_reload(gpu, first, streamed):
    a, b, d = _edges(1, 20_000), _edges(2, 23_000), _edges(3, 11_000)
    with gxp.Context(0) as c:
        c.create_graph(N, 1)
        _load(c, first, *a)
        if first == gxp.GXP_FMT_CSC:
            _check_batch(c, a, streamed)   # makes the host copies
        _load(c, gxp.GXP_FMT_CSC, *b)
        _check_batch(c, b, streamed)
        _load(c, gxp.GXP_FMT_COO, *d)
        _check_batch(c, d, streamed)


@pytest.mark.parametrize("use_graph", [False, True])
@pytest.mark.parametrize("streamed,block_edges", [(False, 0), (True, 0), (True, 100)])
def test_batch_without_edges(gpu, streamed, block_edges, use_graph):
    """A graph without edges: every source reaches itself alone, in one
    superstep that changes nothing; the context goes on with a real graph."""
    none = np.zeros(0, np.uint32)
    a = _edges(4, 5000)
    with gxp.Context(0) as c:
        c.create_graph(N, 1)
        c.load_coo(none, none, none)
        dist, rep = c.sssp_batch(SOURCES, streamed=streamed, block_edges=block_edges, use_graph=use_graph)
        ref = np.full((N, len(SOURCES)), gxp.INF, np.uint32)
        ref[SOURCES, np.arange(len(SOURCES))] = 0
        assert np.array_equal(dist, ref)
        assert rep["supersteps"] == 1
        _load(c, gxp.GXP_FMT_CSC, *a)
        _check_batch(c, a, streamed)
