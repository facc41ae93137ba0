"""Batches around the limits of their default rules: item lengths by the batch's
size and by the shapes that share it, and merging by a query's rows (32,768, or
4,096 from 4 loops on).
Every count equals the same query's run alone, whatever the parameters."""
import numpy as np
import pytest

import datagen

pytestmark = pytest.mark.gpu

OFF = {"merge_min": 0xFFFFFFFF, "merge_ratio": 1}


@pytest.fixture(scope="module")
def hc(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2502_06715_gb300 as hc

    return hc


@pytest.fixture(scope="module")
def graphs(hc):
    """E+ of 60 rows to above 32,768; of exactly that and of 4,096, and a row below."""
    import torch

    eps = [datagen.orient_lt(datagen.rmat_graph(s, ef, 11 + s)) for s, ef in ((5, 4), (9, 8), (12, 8), (13, 9))]
    assert eps[0].shape[0] < 128 and eps[-1].shape[0] > 32768
    eps += [eps[3][:k] for k in (32768, 32767, 4096, 4095)]
    return [hc.build_index(torch.from_numpy(np.ascontiguousarray(e).view(np.int32)).cuda(), 0) for e in eps]


@pytest.mark.parametrize("shapes", ["TRIANGLE", "FOUR_CLIQUE", "TRIANGLE FOUR_CLIQUE", "TRIANGLE FOUR_CLIQUE FOUR_DIAMOND"])
@pytest.mark.parametrize("copies", [1, 40])
def test_default_rules(hc, graphs, shapes, copies):
    import torch

    kinds = [getattr(hc, s) for s in shapes.split()]
    qs, idx = [], []
    for i in range(len(graphs) * copies):
        q = kinds[i % len(kinds)]
        if any(q.attr_order(j) for j in range(len(q.atoms))):
            q = kinds[0]
        qs.append(q)
        idx.append([graphs[i // copies]] * len(q.atoms))
    want = [hc.run_join(q, ix).count for q, ix in zip(qs, idx)]
    side = torch.cuda.Stream()
    for opts in (None, [OFF] * len(qs), [{"merge_min": 32, "merge_ratio": 4}] * len(qs),
                 [{"item_grain": 1 + i % 3} for i in range(len(qs))], [{"dir_min": 0xFFFFFFFF}] * len(qs)):
        b = hc.Batch(qs, idx, opts, stream=side)
        for _ in range(2):
            b.launch(side)
            assert b.counts() == want
        b.free()
