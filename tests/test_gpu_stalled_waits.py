"""Loop 1's and the k-ary sorts' bounded waits that run out, on a GPU, without
faulting it.

Testing flags keep the first tile of loop 1, or of a k-ary sort, from ever
publishing its status word, so the tiles after it wait until the limit, record
the timeout and return.  Every entry point that runs them must then report
HC_ERR_TIMEOUT (4) in bounded time, read nothing that was not written, and
leave the context usable: the next call on the same data is exact.
"""
import contextlib
import time

import numpy as np
import pytest

import datagen
import oracle

pytestmark = pytest.mark.gpu

STALL = 0x100


@pytest.fixture(scope="module")
def hc(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2502_06715_gb300 as hc

    assert hc._lib.HC_FLAG_TEST_STALL_LOOP1 == STALL
    return hc


def dev(rows):
    import torch

    return torch.from_numpy(np.ascontiguousarray(rows, dtype=np.uint32).view(np.int32)).cuda()


@contextlib.contextmanager
def times_out(hc, limit_ns):
    import torch

    prev = hc.set_wait_limit_ns(limit_ns)
    t0 = time.perf_counter()
    try:
        with pytest.raises(hc.HoneycombError) as e:
            yield
    finally:
        hc.set_wait_limit_ns(prev)
    assert e.value.status == 4
    torch.cuda.synchronize()  # no fault is pending on the device
    assert time.perf_counter() - t0 < 20.0


@pytest.fixture(scope="module")
def graph(hc):
    """E+ with about 3,000 first-attribute values (a dozen loop-1 tiles), its index and its triangles."""
    ep = datagen.orient_lt(datagen.rmat_graph(12, 8, 9))
    return hc.build_index(dev(ep), 0), oracle.gj_count(3, list(hc.TRIANGLE.atoms), [ep] * 3)[0], ep


@pytest.mark.parametrize("shares,limit_ns", [([1, 1, 1], 20_000_000), ([1, 1, 1], 0), ([4, 2, 1], 20_000_000)])
def test_join(hc, graph, shares, limit_ns):
    import torch

    ix, want, _ = graph
    with times_out(hc, limit_ns):
        hc.run_join_async(hc.TRIANGLE, [ix] * 3, shares=shares, flags=STALL).count()
    out = torch.empty((want, 3), dtype=torch.int32)
    with times_out(hc, limit_ns):  # single-pass tuples: compaction and copies behind the search
        hc.run_join_to_host(hc.TRIANGLE, [ix] * 3, out, shares=shares, flags=STALL)
    assert hc.run_join(hc.TRIANGLE, [ix] * 3, shares=shares).count == want
    assert hc.run_join_to_host(hc.TRIANGLE, [ix] * 3, out, shares=shares) == want


@pytest.mark.parametrize("stalled", [0, 2])
@pytest.mark.parametrize("mix", ["triangle", "two shapes", "three shapes"])
def test_batch(hc, graph, mix, stalled):
    """One query of a batch stalls: its units are not read, the others' work
    is bounded by theirs, and the batch reports the timeout."""
    import torch

    ix, want, ep = graph
    qs = {"triangle": [hc.TRIANGLE] * 4, "two shapes": [hc.TRIANGLE, hc.FOUR_CLIQUE, hc.TRIANGLE, hc.FOUR_CLIQUE],
          "three shapes": [hc.TRIANGLE, hc.FOUR_CLIQUE, hc.FOUR_CYCLE, hc.TRIANGLE]}[mix]
    side = torch.cuda.Stream()
    idx = [[{o: ix if o == 0 else hc.build_index(dev(ep), 1) for o in (0, 1)}[q.attr_order(j)]
            for j in range(len(q.atoms))] for q in qs]
    good = hc.Batch(qs, idx, stream=side)
    good.launch(side)
    counts = good.counts()
    assert all(c == want for c, q in zip(counts, qs) if q is hc.TRIANGLE)
    for shares in (None, [2, 2] + [1] * (qs[stalled].n_vars - 2)):
        opts = [{} for _ in qs]
        opts[stalled] = {"flags": STALL, **({"shares": shares} if shares else {})}
        bad = hc.Batch(qs, idx, opts, stream=side)
        with times_out(hc, 20_000_000):
            bad.launch(side)
            bad.counts()
        bad.free()
    good.launch(side)  # the memory behind the stalled batch is reused
    assert good.counts() == counts
    good.free()


@pytest.mark.parametrize("limit_ns", [20_000_000, 0])
@pytest.mark.parametrize("shares", [None, (2, 3, 1)])
@pytest.mark.parametrize("wide", [False, True])
def test_kary_build(hc, wide, shares, limit_ns):
    """Packed keys (one sort) and values of 32 bits, which sort a level at a time."""
    rng = np.random.default_rng(3)
    rows = np.unique(rng.integers(0, 90, size=(40_000, 3)).astype(np.uint32), axis=0)
    if wide:
        rows = rows * np.uint32(0x2D00000) + np.uint32(17)
    rows = rows[rng.permutation(rows.shape[0])]
    d = dev(rows)
    kw = {} if shares is None else {"shares": shares, "seeds": (5, 6, 7)}
    with times_out(hc, limit_ns):
        hc.build_kindex(d, test_stall=True, **kw)
    ix = hc.build_kindex(d, **kw)
    assert ix.v(2).shape[0] == rows.shape[0]
    if shares is None:
        want = rows[np.lexsort(rows.T[::-1])]
        assert np.array_equal(ix.v(2).cpu().numpy().view(np.uint32), want[:, 2])
        assert np.array_equal(ix.v(0).cpu().numpy().view(np.uint32), np.unique(rows[:, 0]))
    else:
        got = hc.run_kjoin(hc.KQuery(3, ((0, 1, 2),)), [hc.build_kindex(d)]).count
        assert got == rows.shape[0]


@pytest.mark.parametrize("shares", [[4, 1, 1], [3, 2, 2], [40, 20, 1]])
def test_partitioned_copies(hc, graph, shares):
    """A partitioned copy whose sort gave up has no levels: the join that made
    it must not read them (one and two radix passes, one and three copies)."""
    import torch

    ix, want, _ = graph
    flag = hc._lib.HC_FLAG_TEST_STALL_PARTITION
    with times_out(hc, 20_000_000):
        hc.run_join_async(hc.TRIANGLE, [ix] * 3, shares=shares, flags=flag).count()
    out = torch.empty((want, 3), dtype=torch.int32)
    with times_out(hc, 20_000_000):
        hc.run_join_to_host(hc.TRIANGLE, [ix] * 3, out, shares=shares, flags=flag)
    side = torch.cuda.Stream()
    with times_out(hc, 20_000_000):
        bad = hc.Batch([hc.TRIANGLE] * 2, [[ix] * 3] * 2, [{}, {"shares": shares, "flags": flag}], stream=side)
        bad.launch(side)
        bad.counts()
    assert hc.run_join(hc.TRIANGLE, [ix] * 3, shares=shares).count == want
