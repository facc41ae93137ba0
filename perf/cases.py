"""What a user of this framework has it do, at the sizes they do it at.

    build    CoCo index of a binary relation                      build_index
    join     Generic Join of a built-in query shape, counted or   run_join
             materialized, in one HyperCube cell or many
    view     a join's tuples materialized and indexed as a new    run_join, build_kindex
             ternary relation
    serve    a burst of restricted requests on resident indexes   serve.Server.run
    batch    many queries on many graphs in one launch            Batch
    tensor   Loomis-Whitney over ternary relations, from rows     build_kindex, run_kjoin
             or from resident indexes

Graphs are R-MAT (0.57, 0.19, 0.19, 0.05) with scrambled ids, or uniform;
``E+`` is the relation of the canonical pairs u < v, the symmetric relation
holds both directions.  Everything is drawn on the GPU from the seed; where
the size of a result depends on the graph's shape (an index, tuples, a view),
the shape belongs to the case and the seed draws the ids and the row order.
"""
import math

import numpy as np
import torch

import paper_2502_06715_gb300 as hc
from paper_2502_06715_gb300 import serve

QUERIES = {"triangle": hc.TRIANGLE, "cycle4": hc.FOUR_CYCLE, "diamond": hc.FOUR_DIAMOND, "clique4": hc.FOUR_CLIQUE,
           "two_triangle": hc.TWO_TRIANGLE}
DEV = "cuda"


def listed():
    return [
        # a small graph, one call: an interactive query, bound by launches and host work
        {"name": "triangle_uniform_4k", "kind": "join", "query": "triangle", "graph": "uniform", "scale": 12, "ef": 8,
         "cells": "1,1,1", "mode": "count", "tuned": False},
        # a service's burst of requests, each with a selection of its own, over three resident graphs
        {"name": "serve_rmat20_burst48", "kind": "serve", "scale": 20, "requests": 48, "sample": 16384},
        # an analyst's many small graphs: one replayed launch for 96 triangle and 4-clique counts
        {"name": "batch_96_subgraphs", "kind": "batch", "queries": 96, "edges": 30000},
        # loading the benchmark's graph: 64 M rows, dense ids
        {"name": "build_rmat22", "kind": "build", "graph": "rmat", "scale": 22, "ef": 16, "ids": "dense", "order": 0,
         "drop": 0},
        # loading a relation whose ids are 32-bit hashes, by its second attribute, a ragged size
        {"name": "build_hashed_3m", "kind": "build", "graph": "uniform", "scale": 18, "ef": 12, "ids": "hashed",
         "order": 1, "drop": 40007},
        # the benchmark's query in the benchmark's 64 cells with its tuned schedule, counted per cell: the largest search
        {"name": "triangle_rmat22_64cells", "kind": "join", "query": "triangle", "graph": "rmat", "scale": 22,
         "ef": 16, "cells": "64,1,1", "mode": "count", "tuned": True},
        # all triangles of a mid-size graph written out in a fixed order, the tuned schedule, both attributes partitioned
        {"name": "triangle_rmat19_tuples", "kind": "join", "query": "triangle", "graph": "rmat", "scale": 19,
         "ef": 16, "cells": "4,4,1", "mode": "materialize", "tuned": True},
        # a materialized view: the triangles in one pass, then indexed for the next query
        {"name": "view_rmat17", "kind": "view", "scale": 17, "ef": 16},
        # the deep query of the benchmark, with its intersections rewritten
        {"name": "clique4_rmat17", "kind": "join", "query": "clique4", "graph": "rmat", "scale": 17, "ef": 16,
         "cells": "1,1,1,1", "mode": "count", "tuned": False},
        # closed 4-walks of a symmetric graph: the longest search for its rows
        {"name": "cycle4_rmat13", "kind": "join", "query": "cycle4", "graph": "rmat", "scale": 13, "ef": 16,
         "cells": "1,1,1,1", "mode": "count", "tuned": False},
        # Loomis-Whitney on resident dense tensors
        {"name": "lw_dense_256", "kind": "tensor", "n": 256, "fill": "dense", "spread": 1, "cells": "1,1,1,1",
         "load": False},
        # Loomis-Whitney on sparse tensors, loaded and joined
        {"name": "lw_sparse_200_load", "kind": "tensor", "n": 200, "fill": "sparse", "spread": 5,
         "cells": "1,1,1,1", "load": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "build", "join", "join", "join", "join", "view", "serve", "batch", "tensor", "tensor"])
    if kind == "build":
        scale = rng.randint(10, 21)
        return {"kind": kind, "graph": rng.choice(["rmat", "uniform"]), "scale": scale, "ef": rng.randint(4, 16),
                "ids": rng.choice(["dense", "dense", "hashed"]), "order": rng.randint(0, 1),
                "drop": rng.randint(0, 1 << (scale - 1))}
    if kind == "join":
        q = rng.choice(["triangle", "triangle", "triangle", "cycle4", "diamond", "clique4", "two_triangle"])
        graph = rng.choice(["rmat", "rmat", "uniform"]) if q in ("triangle", "cycle4") else "rmat"
        low, top = {"triangle": (8, 20), "cycle4": (8, 12), "diamond": (8, 12), "clique4": (8, 16),
                    "two_triangle": (8, 10)}[q]
        nv = QUERIES[q].n_vars
        mode = rng.choice(["count", "count", "materialize"]) if q == "triangle" else "count"
        cells = rng.choice([[1] * nv, [1] * nv, [rng.choice([3, 16, 64])] + [1] * (nv - 1),
                            [rng.choice([2, 4]), rng.choice([2, 5])] + [1] * (nv - 2)])
        return {"kind": kind, "query": q, "graph": graph, "scale": rng.randint(low, top),
                "ef": rng.randint(8, 16) if q != "two_triangle" else 8, "cells": ",".join(map(str, cells)),
                "mode": mode, "tuned": mode == "materialize" or rng.random() < 0.3}
    if kind == "view":
        return {"kind": kind, "scale": rng.randint(9, 17), "ef": rng.randint(4, 16)}
    if kind == "serve":
        scale = rng.randint(15, 20)
        return {"kind": kind, "scale": scale, "requests": rng.randint(8, 24),
                "sample": _log(rng, 1 << (scale - 7), 1 << (scale - 5))}
    if kind == "batch":
        return {"kind": kind, "queries": rng.randint(8, 96), "edges": _log(rng, 1000, 60000)}
    if rng.random() < 0.5:
        return {"kind": kind, "n": _log(rng, 48, 256), "fill": "dense", "spread": 1,
                "cells": rng.choice(["1,1,1,1", "1,1,1,1", "2,2,1,2"]), "load": rng.random() < 0.5}
    return {"kind": kind, "n": _log(rng, 64, 200), "fill": "sparse", "spread": rng.randint(3, 5),
            "cells": rng.choice(["1,1,1,1", "1,1,1,1", "2,2,1,2"]), "load": rng.random() < 0.5}


# ------------------------------------------------------------------- inputs

# the schedule the benchmark's autotuner settles on: short work items, no merge path
TUNED = {"item_grain": 16, "merge_min": 0xFFFFFFFF, "merge_ratio": 1}


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed & 0x7FFFFFFFFFFFFFFF)


def _rmat_pairs(scale, m, g):
    """m raw R-MAT edges as (u, v), ids scrambled."""
    u = torch.zeros(m, dtype=torch.int64, device=DEV)
    v = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        r = torch.rand(m, generator=g, device=DEV)
        lower = r >= 0.76
        right = ((r >= 0.57) & (r < 0.76)) | (r >= 0.95)
        u = u * 2 + lower
        v = v * 2 + right
    perm = torch.randperm(1 << scale, generator=g, device=DEV)
    return perm[u], perm[v]


def _edges(graph, scale, ef, g):
    """E+ of the graph: sorted distinct keys u << 32 | v with u < v (int64)."""
    m = ef << scale
    if graph == "rmat":
        u, v = _rmat_pairs(scale, m, g)
    else:
        u = torch.randint(0, 1 << scale, (m,), generator=g, device=DEV)
        v = torch.randint(0, 1 << scale, (m,), generator=g, device=DEV)
    keep = u != v
    u, v = u[keep], v[keep]
    return torch.unique((torch.minimum(u, v) << 32) | torch.maximum(u, v))


def _rows(keys, g):
    """(n, 2) int32 rows of the keys, in a random order."""
    keys = keys[torch.randperm(keys.shape[0], generator=g, device=DEV)]
    return torch.stack([(keys >> 32).to(torch.int32), (keys & 0xFFFFFFFF).to(torch.int32)], dim=1)


def _symmetric(keys):
    return torch.cat([keys, ((keys & 0xFFFFFFFF) << 32) | (keys >> 32)])


def _hash_ids(x, salt):
    """A bijection of 32-bit ids (odd multiplications and shifted xors), as int64."""
    x = ((x ^ salt) * 0x9E3779B1) & 0xFFFFFFFF
    x = x ^ (x >> 15)
    x = (x * 0x85EBCA77) & 0xFFFFFFFF
    return x ^ (x >> 13)


def _relabelled(case, graph, g):
    """The case's own graph, oriented u < v, its ids permuted by the seed: the
    keys first << 32 | second, in no order."""
    keys = _edges(graph, case["scale"], case["ef"], _gen(1000 * case["scale"] + case["ef"]))
    ids = torch.randperm(1 << case["scale"], generator=g, device=DEV)
    return (ids[keys >> 32] << 32) | ids[keys & 0xFFFFFFFF]


def _build_rows(case, seed):
    g = _gen(seed)
    keys = _edges(case["graph"], case["scale"], case["ef"], _gen(1000 * case["scale"] + case["ef"]))
    keys = keys[torch.randperm(keys.shape[0], generator=_gen(case["scale"]), device=DEV)]
    keys = keys[: max(1, keys.shape[0] - case["drop"])]
    hi, lo = keys >> 32, keys & 0xFFFFFFFF
    if case["ids"] == "hashed":
        salt = int(torch.randint(0, 1 << 32, (1,), generator=g, device=DEV).item())
        hi, lo = _hash_ids(hi, salt), _hash_ids(lo, salt)
    else:
        ids = torch.randperm(1 << case["scale"], generator=g, device=DEV)
        hi, lo = ids[hi], ids[lo]
    order = torch.randperm(keys.shape[0], generator=g, device=DEV)
    to32 = lambda t: torch.where(t > 0x7FFFFFFF, t - (1 << 32), t).to(torch.int32)  # noqa: E731
    return torch.stack([to32(hi[order]), to32(lo[order])], dim=1)


def _cells(case):
    return [int(x) for x in case["cells"].split(",")]


def _tensor_rows(case, seed):
    """The four ternary relations of LW.  dense: a box [a] x [b] x [c] whose
    sides are within an eighth of n; sparse: about n^3 distinct rows of [spread n]^3."""
    g = _gen(seed)
    n = case["n"]
    out = []
    for _ in range(4):
        if case["fill"] == "dense":
            a, b, c = (int(x) for x in torch.randint(n - n // 8, n + 1, (3,), generator=g, device=DEV).tolist())
            keys = torch.arange(a * b * c, device=DEV)
            x, y, z = keys // (b * c), keys // c % b, keys % c
        else:
            d = case["spread"] * n
            keys = torch.unique(torch.randint(0, d ** 3, (n ** 3,), generator=g, device=DEV))
            x, y, z = keys // (d * d), keys // d % d, keys % d
        rows = torch.stack([x, y, z], dim=1).to(torch.int32)
        out.append(rows[torch.randperm(rows.shape[0], generator=g, device=DEV)].contiguous())
    return out


def _build_tensors(case, rels):
    cells = _cells(case)
    if max(cells) == 1:
        return [hc.build_kindex(r, hc.LW.level_cols(j)) for j, r in enumerate(rels)]
    per_atom = hc.atom_shares(hc.LW, cells)
    return [hc.build_kindex(r, hc.LW.level_cols(j), seeds=per_atom[j][0], shares=per_atom[j][1])
            for j, r in enumerate(rels)]


def _graph_indexes(query, keys, g):
    """One index per atom of the query over one relation (an index per attribute order)."""
    rows = _rows(keys, g)
    by_order = {o: hc.build_index(rows, o) for o in {query.attr_order(j) for j in range(len(query.atoms))}}
    return [by_order[query.attr_order(j)] for j in range(len(query.atoms))]


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    g = _gen(seed)
    if kind == "build":
        st["rows"] = _build_rows(case, seed)
    elif kind == "join":
        q = QUERIES[case["query"]]
        keys = _relabelled(case, case["graph"], g) if case["mode"] == "materialize" else \
            _edges(case["graph"], case["scale"], case["ef"], g)
        if case["query"] == "cycle4":
            keys = _symmetric(keys)
        st["query"], st["indexes"] = q, _graph_indexes(q, keys, g)
    elif kind == "view":
        st["indexes"] = _graph_indexes(hc.TRIANGLE, _relabelled(case, "rmat", g), g)
        # the room for the tuples, from a count when the view was planned
        st["capacity"] = int(1.25 * hc.run_join(hc.TRIANGLE, st["indexes"]).count) + 1
    elif kind == "serve":
        s = case["scale"]
        rmat = _symmetric(_edges("rmat", s, 16, g))
        rels = {"rmat": rmat, "uniform_a": _symmetric(_edges("uniform", s, 8, g)),
                "uniform_b": _symmetric(_edges("uniform", s, 2, g))}
        st["server"] = serve.Server({k: hc.build_index(_rows(v, g)) for k, v in rels.items()})
        # requests select among vertices of ordinary degree
        degree = torch.bincount(rmat >> 32, minlength=1 << s)
        ordinary = torch.nonzero((degree > 0) & (degree <= 64)).reshape(-1).cpu().numpy().astype(np.uint32)
        rng = np.random.default_rng(seed)
        names = sorted(rels)
        shapes = [hc.TRIANGLE, hc.TRIANGLE, hc.FOUR_CYCLE]
        st["requests"] = []
        for i in range(case["requests"]):
            q = shapes[int(rng.integers(len(shapes)))]
            size = min(ordinary.shape[0], int(case["sample"] * 2.0 ** rng.uniform(-1.0, 1.0)))
            pick = rng.choice(ordinary, size=max(1, size), replace=False)
            st["requests"].append(serve.Request(i, q.with_atoms([(v, None) for v in range(q.n_vars)]),
                                                tuple(names[int(k)] for k in rng.integers(3, size=len(q.atoms))), pick))
    elif kind == "batch":
        rng = np.random.default_rng(seed)
        queries, indexes = [], []
        for _ in range(case["queries"]):
            q = hc.TRIANGLE if rng.random() < 0.5 else hc.FOUR_CLIQUE
            edges = case["edges"] * 4.0 ** rng.uniform(-1.0, 1.0)
            scale = max(7, int(math.log2(edges / 8)))
            keys = _edges("rmat", scale, max(1, int(edges / (1 << scale))), g)
            queries.append(q)
            indexes.append(_graph_indexes(q, keys, g))
        st["stream"] = torch.cuda.Stream()
        st["batch"] = hc.Batch(queries, indexes, stream=st["stream"])
        st["batch"].capture(st["stream"])
        st["keep"] = indexes
    else:
        rels = _tensor_rows(case, seed)
        if case["load"]:
            st["rows"] = rels
        else:
            st["indexes"] = _build_tensors(case, rels)
    return st


# -------------------------------------------------------------------- calls

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "build":
        ix = hc.build_index(st["rows"], case["order"])
        return {"keys": ix.keys(), "v1": ix.v1(), "o1": ix.o1(), "v2": ix.v2()}
    if kind == "join":
        many = max(_cells(case)) > 1
        r = hc.run_join(st["query"], st["indexes"], shares=_cells(case), mode=case["mode"], cell_counts=many,
                        keep_device=True, **(TUNED if case["tuned"] else {}))
        out = {"count": r.count}
        if many:
            out["cells"] = r.cell_counts
        if case["mode"] == "materialize":
            out["tuples"] = r.tuples
        return out
    if kind == "view":
        r = hc.run_join(hc.TRIANGLE, st["indexes"], mode="materialize", out_capacity=st["capacity"], keep_device=True)
        ix = hc.build_kindex(r.tuples)
        return {"count": r.count, "v0": ix.v(0), "o0": ix.o(0), "v1": ix.v(1), "o1": ix.o(1), "v2": ix.v(2)}
    if kind == "serve":
        done = st["server"].run(st["requests"], realtime=False)
        return np.array([o.count for o in sorted(done, key=lambda o: o.rid)], dtype=np.int64)
    if kind == "batch":
        st["batch"].launch(st["stream"])
        return np.array(st["batch"].counts(), dtype=np.int64)
    indexes = st["indexes"] if "indexes" in st else _build_tensors(case, st["rows"])
    many = max(_cells(case)) > 1
    r = hc.run_kjoin(hc.LW, indexes, cell_counts=many)
    return {"count": r.count, "cells": r.cell_counts} if many else {"count": r.count}


# --------------------------------------------------------------------- sizes

def _n_edges(graph, scale, ef):
    """Expected rows of E+: the distinct ones of ef * 2^scale draws."""
    m = float(ef << scale)
    if graph == "uniform":
        space = 2.0 ** (2 * scale - 1)
        return space * (1.0 - math.exp(-m / space))
    return m * max(0.4, 1.0 - 0.035 * max(0, 23 - scale) * ef / 16)


def _n_triangles(scale, ef):
    """Triangles of the R-MAT graph: about 2.1e9 at scale 22 and edge factor 16, 2.35 times more a scale."""
    return 2.1e9 * 2.35 ** (scale - 22) * (ef / 16) ** 2.2


def work(case):
    """Relations (or the levels of their indexes) read once, results written once."""
    kind = case["kind"]
    if kind == "build":
        n = max(1.0, _n_edges(case["graph"], case["scale"], case["ef"]) - case["drop"])
        return {"bytes": n * (8 + 8 + 4) + 8 * min(n, 2.0 ** case["scale"]), "flops": 0}
    if kind == "join":
        n = _n_edges(case["graph"], case["scale"], case["ef"]) * (2 if case["query"] == "cycle4" else 1)
        out = 12 * _n_triangles(case["scale"], case["ef"]) if case["mode"] == "materialize" else 0
        return {"bytes": 4 * n + 8 * min(n, 2.0 ** case["scale"]) + out, "flops": 0}
    if kind == "view":
        n, t = _n_edges("rmat", case["scale"], case["ef"]), _n_triangles(case["scale"], case["ef"])
        return {"bytes": 4 * n + 8 * 2.0 ** case["scale"] + 4 * t + 8 * n, "flops": 0}
    if kind == "serve":
        return {"bytes": case["requests"] * case["sample"] * 4 * (1 + 16.0), "flops": 0}
    if kind == "batch":
        return {"bytes": case["queries"] * case["edges"] * 5.0, "flops": 0}
    rows = 4.0 * case["n"] ** 3
    return {"bytes": rows * (12 if case["load"] else 4), "flops": 0}


# ---------------------------------------------------------------------- exact

def exact(case, seed):
    kind = case["kind"]
    if kind == "build":
        rows = _build_rows(case, seed).to(torch.int64) & 0xFFFFFFFF
        a, b = (rows[:, 1], rows[:, 0]) if case["order"] else (rows[:, 0], rows[:, 1])
        # sort as unsigned: flip the top bit of the packed key
        top = torch.iinfo(torch.int64).min
        keys = torch.sort(((a << 32) | b) ^ top).values ^ top
        hi, lo = (keys >> 32) & 0xFFFFFFFF, keys & 0xFFFFFFFF
        v1, counts = torch.unique_consecutive(hi, return_counts=True)
        o1 = torch.cat([counts.new_zeros(1), counts.cumsum(0)])
        return {"keys": keys, "v1": v1.to(torch.int32), "o1": o1.to(torch.int32), "v2": lo.to(torch.int32)}
    if kind == "join" and case["query"] == "triangle" and case["mode"] == "count" and max(_cells(case)) == 1 \
            and case["scale"] <= 13:
        keys = _edges(case["graph"], case["scale"], case["ef"], _gen(seed))
        u, v = keys >> 32, keys & 0xFFFFFFFF
        adj = torch.zeros(1 << case["scale"], 1 << case["scale"], dtype=torch.float64, device=DEV)
        adj[u, v] = 1.0
        return {"count": int((adj @ adj)[u, v].sum().item())}
    if kind == "tensor" and case["fill"] == "dense" and max(_cells(case)) == 1:
        sides = [tuple(int(x) + 1 for x in r.max(dim=0).values.tolist()) for r in _tensor_rows(case, seed)]
        count = 1
        for var in range(4):
            count *= min(s[a.index(var)] for s, a in zip(sides, hc.LW.atoms) if var in a)
        return {"count": count}
    return None
