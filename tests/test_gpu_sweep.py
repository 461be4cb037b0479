"""The single-partition superstep kernel at the edges of its work items:
rows whose in-degrees sit at the borders of the lane groups (1..32 lanes a
row), the narrow-slice groups and the hub parts, with each number of columns
the layout aims at (it follows the edge count), vertices inside and past the
staged values, renumbered or not; and two contexts running at once, whose
persistent kernels share the GPU. Against the oracle: SSSP and CC bit for
bit, PageRank and personalized PageRank within the fp32 bars of the other
superstep tests (relative 1e-4, L1 1e-5)."""
import threading

import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu

DEGREES = [0, 1, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257,
           511, 512, 513, 1024, 2047, 2048, 2049, 4097, 9001]


def _graph(n, extra, seed):
    """Rows of the listed in-degrees (a few of each, at scattered ids) and
    `extra` edges whose destinations crowd at the low ids, so that in-degrees
    of every size occur; sources uniform, weights U{1..100}."""
    rng = np.random.default_rng(seed)
    rows = rng.permutation(n)[: 5 * len(DEGREES)]
    deg = np.repeat(DEGREES, 5)
    dst = np.concatenate([np.repeat(rows, deg), (n * rng.random(extra) ** 3).astype(np.int64)]).astype(np.uint32)
    src = rng.integers(0, n, len(dst)).astype(np.uint32)
    return src, dst, rng.integers(1, 101, len(dst)).astype(np.uint32)


def _check_ranks(r, ref):
    r = r.astype(np.float64)
    nz = ref > 0
    assert np.all(r[~nz] == 0)
    assert (np.abs(r - ref)[nz] / ref[nz]).max() <= 1e-4
    assert np.abs(r - ref).sum() <= 1e-5


# extra edges: 4, 8 and 16 columns a lane (borders at 2^21 and 2^23 edges);
# vertices: all values staged, one past the staged 32,768, and many past it
@pytest.mark.parametrize("n,extra", [(257, 0), (32767, 1000), (32768, 100_000), (40_000, 2_200_000),
                                     (300_001, 8_500_000)])
@pytest.mark.parametrize("keep_ids", [False, True])
def test_rows_at_item_borders(n, extra, keep_ids):
    src, dst, w = _graph(n, extra, n)
    source = int(src[0])
    d_ref, steps, _ = oracle.sssp(n, src, dst, w, source)
    l_ref, l_steps, _ = oracle.cc(n, src, dst)
    r_ref, _, _ = oracle.pagerank(n, src, dst, 0.85, 6)
    with gxp.Context(0, keep_ids=keep_ids) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst, w)
        assert c.run(gxp.GXP_ALGO_SSSP, source) == steps
        assert np.array_equal(c.values(), d_ref)
        assert c.run(gxp.GXP_ALGO_CC) == l_steps
        assert np.array_equal(c.values(), l_ref)
        c.run(gxp.GXP_ALGO_PAGERANK, max_steps=6)
        whole = c.values()
        _check_ranks(whole, r_ref)
        c.begin(gxp.GXP_ALGO_PAGERANK)   # a launch per superstep: the same bits
        for _ in range(6):
            c.superstep(want_changed=False)
        assert np.array_equal(c.values(), whole)


@pytest.mark.parametrize("direction", [gxp.GXP_DIR_AUTO, gxp.GXP_DIR_PULL, gxp.GXP_DIR_PUSH])
def test_low_timeout_takes_a_launch_per_superstep(direction):
    """A limit on device waits below the default runs without any: the same
    results, no persistent launch."""
    n = 5000
    src, dst, w = _graph(n, 20_000, 9)
    d_ref, steps, _ = oracle.sssp(n, src, dst, w, 3)
    r_ref, _, _ = oracle.pagerank(n, src, dst, 0.85, 4)
    with gxp.Context(0, timeout_ns=1000, direction=direction) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst, w)
        assert c.run(gxp.GXP_ALGO_SSSP, 3) == steps
        assert np.array_equal(c.values(), d_ref)
        assert c.stats()["persistent_launches"] == 0
        assert c.run(gxp.GXP_ALGO_PAGERANK, max_steps=4) == 4
        _check_ranks(c.values(), r_ref)


def test_two_contexts_at_once():
    """Persistent kernels of two contexts, driven by two threads, take turns
    on the GPU: every run of both gives the oracle's results."""
    n = 60_000
    src, dst, w = _graph(n, 400_000, 5)
    d_ref, steps, _ = oracle.sssp(n, src, dst, w, 1)
    r_ref, _, _ = oracle.pagerank(n, src, dst, 0.85, 20)
    errors = []

    def work(which):
        try:
            with gxp.Context(0) as c:
                c.create_graph(n, 1)
                c.load_coo(src, dst, w)
                for _ in range(20):
                    if which:
                        assert c.run(gxp.GXP_ALGO_SSSP, 1) == steps
                        assert np.array_equal(c.values(), d_ref)
                    else:
                        c.run(gxp.GXP_ALGO_PAGERANK, max_steps=20)
                        _check_ranks(c.values(), r_ref)
        except BaseException as e:   # noqa: BLE001 - handed to the test's thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
