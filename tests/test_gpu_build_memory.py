"""The device memory a build holds at its peak and keeps.

A build holds 20 bytes a row of keys and levels, 16 of directory, asked for
ahead, and, until it is done, about 8.4 of scratch.  An index without a
run of 16 values or more gives the directory's block back.  Read from the
device's default memory pool through the driver."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

USED_NOW, USED_HIGH = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH


@pytest.fixture(scope="module")
def hc(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2502_06715_gb300 as hc

    return hc


class Pool:
    def __init__(self):
        self.cu = ctypes.CDLL("libcuda.so.1")
        dev, self.pool = ctypes.c_int(), ctypes.c_void_p()
        assert self.cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.pool), dev) == 0

    def get(self, attr):
        v = ctypes.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.pool, attr, ctypes.byref(v)) == 0
        return v.value

    def reset_high(self):
        assert self.cu.cuMemPoolSetAttribute(self.pool, USED_HIGH, ctypes.byref(ctypes.c_uint64(0))) == 0


@pytest.mark.parametrize("run", [1, 8, 15, 16, 40])
@pytest.mark.parametrize("n", [15, 16, 6145, 1_000_003])
def test_peak_and_kept(hc, n, run):
    import torch

    k = np.arange(n, dtype=np.uint32)
    rows = np.stack([k // run * 3, k % run * 7], axis=1)[np.random.default_rng(n).permutation(n)]
    d = torch.from_numpy(np.ascontiguousarray(rows, dtype=np.uint32).view(np.int32)).cuda()
    torch.cuda.synchronize()
    pool = Pool()
    before = pool.get(USED_NOW)
    pool.reset_high()
    ix = hc.build_index(d, 0)
    torch.cuda.synchronize()
    slack = 64 * 1024
    v1pos = 4 * ix._view.v1pos_n
    assert pool.get(USED_HIGH) - before <= 44.4 * n + v1pos + slack
    longest = min(n, run)
    kept = 20 * n + (16 * n if longest >= 16 else 0) + v1pos + (16 * ix.l1 if v1pos == 0 and ix.l1 >= 16 else 0)
    assert pool.get(USED_NOW) - before <= kept + slack
    assert np.array_equal(ix.v1().cpu().numpy().view(np.uint32), np.unique(rows[:, 0]))
    order = np.lexsort((rows[:, 1], rows[:, 0]))
    assert np.array_equal(ix.v2().cpu().numpy().view(np.uint32), rows[order, 1])
    ix.free()
    torch.cuda.synchronize()
    assert pool.get(USED_NOW) <= before + slack
