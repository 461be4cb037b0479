"""gxp_get_values into device memory: whole tensors and views at an offset; an
array that ends before n values is refused by the host, before anything is
written."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2203_13005_gb300 import gxp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1000, 3 << 20])
def test_device_arrays(gpu, n):
    import torch
    rng = np.random.default_rng(2)
    src, dst = rng.integers(0, n, 2 * n).astype(np.uint32), rng.integers(0, n, 2 * n).astype(np.uint32)
    ref, _, _ = oracle.cc(n, src, dst)
    with gxp.Context(0) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst)
        c.run(gxp.GXP_ALGO_CC)
        out = torch.zeros(n, dtype=torch.int32, device="cuda")
        c.values(out=out)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), ref)
        big = torch.full((n + 9,), 7, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        c.values(out=big[5:5 + n])
        got = big.cpu().numpy().view(np.uint32)
        assert np.array_equal(got[5:5 + n], ref) and np.all(got[:5] == 7) and np.all(got[5 + n:] == 7)


def test_array_too_small(gpu):
    import torch
    n = 3 << 20
    src, dst = np.arange(n - 1, dtype=np.uint32), np.arange(1, n, dtype=np.uint32)
    with gxp.Context(0) as c:
        c.create_graph(n, 1)
        c.load_coo(src, dst)
        c.run(gxp.GXP_ALGO_PAGERANK, max_steps=1)
        torch.cuda.empty_cache()
        # 32 MB, a device allocation of its own, whose tail is shorter than n values
        block = torch.full((8 << 20,), 3, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        tail = block[(8 << 20) - 1000:]
        rc = c.lib.gxp_get_values(c.h, gxp.ALL_PARTS, ctypes.c_void_p(tail.data_ptr()), n)
        assert rc == gxp.GXP_E_INVAL
        assert int((block != 3).sum()) == 0
        assert abs(float(c.values().sum()) - 1.0) < 1e-3   # not poisoned
