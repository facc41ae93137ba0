"""The order of two-pass tuples is fixed by the call, not by the launch.

The work items decide the order in which tuples come out.  With item_grain 0
the library cuts them by the join's size; the cut must not follow the number
of warps that happen to run (block_threads sets it: 32 warps an SM with one
warp a block, 64 with four), or the same call would give another order on
another device.
"""
import numpy as np
import pytest

import datagen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hc(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2502_06715_gb300 as hc

    return hc


@pytest.mark.parametrize("shares", [[1, 1, 1], [3, 2, 1]])
def test_default_order_does_not_follow_the_launch(hc, shares):
    import torch

    ep = datagen.orient_lt(datagen.rmat_graph(15, 16, 5))
    d = torch.from_numpy(np.ascontiguousarray(ep).view(np.int32)).cuda()
    ix = hc.build_index(d, 0)
    want = oracle.gj_count(3, list(hc.TRIANGLE.atoms), [ep] * 3)[0]
    runs = [hc.run_join(hc.TRIANGLE, [ix] * 3, shares=shares, mode="materialize", block_threads=bt)
            for bt in (128, 32, 96, 0)]
    for r in runs:
        assert r.count == want and r.tuples.shape[0] == want
        assert r.n_items == runs[0].n_items
        assert torch.equal(r.tuples, runs[0].tuples)
