"""k-ary counting over dense last-loop lists of any length.

Dense lists are kept as bitmaps and a binding whose last-loop lists are all
dense is counted from the words' AND: by one lane when a batch has many
bindings, by the whole warp when it has few long ones, and through the
per-binding search past 512 words (16,384 values of span).  The sizes lie
around those limits; the expected counts come from numpy.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hc(cuda_device):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2502_06715_gb300 as hc

    return hc


def dev(rows):
    import torch

    return torch.from_numpy(np.ascontiguousarray(rows, dtype=np.uint32).view(np.int32)).cuda()


def _rows(mask, base):
    """Ternary rows (a, b, base + u) of a boolean array indexed [a][b][u]."""
    a, b, u = np.nonzero(mask)
    return np.stack([a, b, u + base], axis=1).astype(np.uint32)


@pytest.mark.parametrize("base", [0, 45])
@pytest.mark.parametrize("span", [33, 1100, 16352, 16384, 16417, 40000])
@pytest.mark.parametrize("nx,ny,nz", [(2, 2, 1), (2, 2, 5), (1, 3, 40)])
def test_lists_of_every_length(hc, span, nx, ny, nz, base):
    """Q(x, y, z, u) <- A(x, y, z), R(x, y, u), S(x, z, u), T(y, z, u): up to
    nz bindings in a batch, each intersecting three lists of about span / 2
    values; one list of each relation is sparse, so some bindings search."""
    rng = np.random.default_rng(1000 * span + 10 * nz + base)
    masks = []
    for na, nb in ((nx, ny), (nx, nz), (ny, nz)):
        m = rng.random((na, nb, span)) < 0.5
        m[-1, -1] = rng.random(span) < 0.02  # a sparse list among dense ones
        m[..., 0] = m[..., -1] = True
        masks.append(m)
    r, s, t = masks
    want = int(np.einsum("xyu,xzu,yzu->", r.astype(np.int64), s.astype(np.int64), t.astype(np.int64), optimize=True))
    a = np.stack(np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"), -1).reshape(-1, 3)
    q = hc.KQuery(4, ((0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3)))
    rels = [a, _rows(r, base), _rows(s, base), _rows(t, base)]
    ixs = [hc.build_kindex(dev(x), q.level_cols(j)) for j, x in enumerate(rels)]
    for kw in ({}, {"pair_min": 0xFFFFFFFF}, {"item_grain": 1}):
        assert hc.run_kjoin(q, ixs, **kw).count == want, kw
    cells = hc.run_kjoin(q, ixs, cell_counts=True)
    assert int(cells.cell_counts.sum().item()) == want


def test_single_dense_list(hc):
    """A last loop of one dense list: every value of it is a result."""
    rng = np.random.default_rng(8)
    m = rng.random((1, 70, 9000)) < 0.5
    s = _rows(m, 3)[:, 1:]
    e = np.stack([np.arange(200), rng.integers(0, 70, 200)], axis=1)
    want = int(m[0][e[:, 1]].sum())
    q = hc.KQuery(3, ((0, 1), (1, 2)))
    ixs = [hc.build_kindex(dev(e), q.level_cols(0)), hc.build_kindex(dev(s), q.level_cols(1))]
    assert hc.run_kjoin(q, ixs).count == want
