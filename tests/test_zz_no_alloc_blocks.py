"""Edge-block sizes of the allocation-free superstep (gxp_superstep_min_noalloc),
collected last like the entry point's other tests."""
import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp
from test_zz_no_alloc import _csc, _noalloc, _padded_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 64, 5000, 200_000])
@pytest.mark.parametrize("hub", [0, 15, 17, 65, 513, 70_000])
def test_noalloc_block_sizes(n, hub):
    """Edge blocks of every size the call picks (64 to 2048 merge items, by
    the input's size) with rows at and over a block's split limit, against
    the oracle's superstep."""
    rng = np.random.default_rng(n + hub)
    m = 12 * n
    dst = np.concatenate([rng.integers(0, n, m), np.full(hub, n // 2)]).astype(np.uint32)
    src = rng.integers(0, n, len(dst)).astype(np.uint32)
    w = rng.integers(1, 101, len(dst)).astype(np.uint32)
    col_ptr, csrc, cw = _csc(n, src, dst, w)
    d_cp, d_src, d_w = _padded_device(col_ptr), _padded_device(csrc), _padded_device(cw)
    cur = rng.integers(0, 1000, n).astype(np.uint32)
    cur[rng.random(n) < 0.5] = gxp.INF
    d_a = _padded_device(cur)
    import torch
    d_b = torch.zeros_like(d_a)
    for algo, step, wt in ((gxp.GXP_ALGO_SSSP, lambda: oracle.sssp_step(n, src, dst, w, cur), d_w),
                           (gxp.GXP_ALGO_CC, lambda: oracle.cc_step(n, src, dst, cur), None)):
        ref, rch = step()
        ch = _noalloc(algo, n, len(src), d_cp, d_src, wt, d_a, d_b)
        assert ch == rch
        assert np.array_equal(d_b[:n].cpu().numpy().view(np.uint32), ref)
