"""Performance cases of the sparse-product library, and their inputs.

A case is a dict of plain values; ``op`` names the public call it stands for:

* ``spgemm``    -- ``sg.spgemm(A, A)``, the whole product from CSR to CSR;
* ``masked``    -- ``sg.masked_spgemm(A, A, A)``, the product inside A's pattern
  (triangle counting on integer values);
* ``kslice``    -- ``sg.spgemm_kslice(A, A, c)``: c slices of the inner dimension
  multiplied one by one, then merged;
* ``merge``     -- ``sg.merge(parts)``: the sum of c partial products that are in
  hand already (what a rank does after it has received them);
* ``batch``     -- many uneven products with one plan (plan, symbolic, numeric);
* ``galerkin``  -- a kept ``GalerkinChain``, replayed on its operators: the setup of
  a multigrid hierarchy, as a captured graph of launches or as one persistent
  launch;
* ``mcl``       -- ``sg.mcl_step`` with the trained row-size predictor: a Markov
  clustering expansion, pruned and renormalised;
* ``transpose`` -- ``sg.transpose(A)``.

Inputs are made on the GPU.  A case fixes its graph up to the names of the
vertices, and the seed draws these and the values: products of other seeds
have other rows, columns and values, and as many entries.  Graphs are R-MAT
with the Graph500 quadrant probabilities, symmetrised, of any order (the first
n vertices of a shuffled power of two); Erdos-Renyi matrices have about d
entries per column; grids are 7-point stencils with random coefficients,
aggregated 2 x 2 x 2.
"""
from __future__ import annotations

import math
import zlib

import numpy as np
import torch

from paper_1510_00844_gb300 import amg
from paper_1510_00844_gb300 import spgemm as sg

DEV = "cuda"
G500 = (0.57, 0.19, 0.19)
THRESHOLD = 1e-4
MARGIN = 0.35
VALUE_DTYPES = {"f64": torch.float64, "f32": torch.float32, "i64": torch.int64, "none": None}
INDEX_DTYPES = {"i32": torch.int32, "i64": torch.int64}


# ------------------------------------------------------------------ cases
def listed():
    return [
        # a small graph: the latency of one call, every phase and its launches
        {"name": "graph_1k", "op": "spgemm", "graph": "rmat", "n": 1000, "d": 16,
         "value": "f64", "index": "i32"},
        # Erdos-Renyi, 8 per column: short rows only, no skew
        {"name": "er_16k", "op": "spgemm", "graph": "er", "n": 16384, "d": 8,
         "value": "f64", "index": "i32"},
        # triangle counts of an ordinary graph: integers, 64-bit indices, a mask
        {"name": "triangles_30k", "op": "masked", "graph": "rmat", "n": 30011, "d": 16,
         "value": "i64", "index": "i64"},
        # two-hop reachability: the pattern alone
        {"name": "reach_100k", "op": "spgemm", "graph": "rmat", "n": 100003, "d": 8,
         "value": "none", "index": "i32"},
        # Graph500 squaring at scale 18, the largest product
        {"name": "graph_262k", "op": "spgemm", "graph": "rmat", "n": 262144, "d": 16,
         "value": "f64", "index": "i32"},
        # the inner dimension in four slices, and their merge
        {"name": "kslice4_65k", "op": "kslice", "graph": "rmat", "n": 65536, "d": 16, "c": 4,
         "value": "f64", "index": "i32"},
        # four partial products received by one rank: the merge alone
        {"name": "merge4_100k", "op": "merge", "n": 100003, "d": 384, "c": 4, "value": "f64",
         "index": "i32"},
        # uneven independent products in single precision
        {"name": "batch_64", "op": "batch", "count": 64, "nmin": 1024, "nmax": 65536, "dmin": 4,
         "dmax": 32, "value": "f32", "index": "i32"},
        # three Galerkin levels of a 128^3 grid, with their transposes, as one graph
        {"name": "galerkin_128", "op": "galerkin", "nx": 128, "ny": 128, "nz": 128, "levels": 3,
         "persistent": False},
        # the same hierarchy of a smaller, uneven grid in one persistent launch
        {"name": "galerkin_50_persistent", "op": "galerkin", "nx": 50, "ny": 64, "nz": 47,
         "levels": 3, "persistent": True},
        # one Markov clustering step with learned sizing
        {"name": "mcl_40k", "op": "mcl", "n": 40009, "d": 16, "index": "i32"},
        # a transpose with the long rows of a power-law graph
        {"name": "transpose_262k", "op": "transpose", "graph": "rmat", "n": 262144, "d": 16,
         "value": "f64", "index": "i32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case; its sizes stay below those of the largest listed case."""
    op = rng.choice(["spgemm", "spgemm", "spgemm", "masked", "kslice", "merge", "batch", "galerkin",
                     "mcl", "transpose"])
    index = rng.choice(["i32", "i32", "i64"])
    if op == "spgemm":
        graph = rng.choice(["rmat", "rmat", "er"])
        return {"op": op, "graph": graph, "n": _log(rng, 700, 180000), "d": rng.randint(4, 16),
                "value": rng.choice(["f64", "f64", "f32", "i64", "none"]), "index": index}
    if op == "masked":
        return {"op": op, "graph": rng.choice(["rmat", "er"]), "n": _log(rng, 1500, 50000),
                "d": rng.randint(4, 16), "value": rng.choice(["i64", "f64"]), "index": index}
    if op == "kslice":
        return {"op": op, "graph": rng.choice(["rmat", "rmat", "er"]), "n": _log(rng, 3000, 60000),
                "d": rng.randint(6, 16), "c": rng.randint(2, 10),
                "value": rng.choice(["f64", "f32", "i64"]), "index": index}
    if op == "merge":
        return {"op": op, "n": _log(rng, 4000, 90000), "d": rng.randint(16, 160),
                "c": rng.randint(2, 9), "value": rng.choice(["f64", "f64", "f32", "none"]),
                "index": index}
    if op == "batch":
        return {"op": op, "count": _log(rng, 6, 96), "nmin": rng.choice([256, 1024]),
                "nmax": _log(rng, 4096, 65536), "dmin": 4, "dmax": rng.randint(8, 32),
                "value": rng.choice(["f32", "f32", "f64", "none"]), "index": index}
    if op == "galerkin":
        levels = rng.randint(1, 3)
        return {"op": op, "nx": rng.randint(16, 120), "ny": rng.randint(16, 120),
                "nz": rng.randint(16, 120), "levels": levels,
                "persistent": rng.random() < 0.5}
    if op == "mcl":
        return {"op": op, "n": _log(rng, 2000, 50000), "d": rng.randint(6, 16), "index": index}
    return {"op": op, "graph": rng.choice(["rmat", "er"]), "n": _log(rng, 1000, 262144),
            "d": rng.randint(4, 16), "value": rng.choice(["f64", "f32", "none"]), "index": index}


# ----------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _own_generator(case):
    """The generator of what a case fixes for every seed."""
    text = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    return _generator(zlib.crc32(text.encode()))


def _shuffle(gen, n):
    return torch.randperm(n, generator=gen, device=DEV)


def _values(gen, nnz, value):
    if value == "f64":
        return torch.rand(nnz, generator=gen, device=DEV, dtype=torch.float64)
    if value == "f32":
        return torch.rand(nnz, generator=gen, device=DEV, dtype=torch.float32) * 2 - 1
    if value == "i64":
        return torch.randint(-3, 4, (nnz,), generator=gen, device=DEV)
    return None


def _csr(nrows, ncols, keys, index, val):
    """CSR of the ascending, distinct keys row * ncols + col."""
    rows = keys // ncols
    rowptr = torch.zeros(nrows + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.bincount(rows, minlength=nrows).cumsum(0)
    return sg.DeviceCSR(nrows, ncols, rowptr, (keys - rows * ncols).to(INDEX_DTYPES[index]), val)


def _rmat_keys(gen, n, d):
    """Distinct keys of a symmetrised R-MAT graph of about d edges per vertex,
    restricted to n of its vertices."""
    scale = max(1, (n - 1).bit_length())
    full = 1 << scale
    edges = d * full
    a, b, c = G500
    src = torch.zeros(edges, dtype=torch.int64, device=DEV)
    dst = torch.zeros(edges, dtype=torch.int64, device=DEV)
    for bit in range(scale):
        r = torch.rand(edges, generator=gen, device=DEV)
        src |= (r >= a + b).to(torch.int64) << bit
        dst |= (((r >= a) & (r < a + b)) | (r >= a + b + c)).to(torch.int64) << bit
    if n < full:
        perm = _shuffle(gen, full)
        src, dst = perm[src], perm[dst]
        keep = (src < n) & (dst < n)
        src, dst = src[keep], dst[keep]
    return torch.unique(torch.cat([src * n + dst, dst * n + src]))


def _er_keys(gen, n, d):
    rows = torch.randint(0, n, (n, d), generator=gen, device=DEV)
    cols = torch.arange(n, device=DEV)[:, None]
    return torch.unique((rows * n + cols).reshape(-1))


def _keys(gen, case):
    kind = _rmat_keys if case.get("graph", "rmat") == "rmat" else _er_keys
    return kind(gen, case["n"], case["d"])


def _relabelled(keys, n, rows, cols):
    return rows[keys // n] * n + cols[keys % n]


def _matrix(own, gen, case, rows, cols):
    """The case's next matrix with its rows and columns renamed."""
    n = case["n"]
    keys = torch.sort(_relabelled(_keys(own, case), n, rows, cols)).values
    return _csr(n, n, keys, case["index"], _values(gen, keys.numel(), case["value"]))


def _markov(own, gen, n, d, index):
    """Rows of M^T: a graph with a self loop on every vertex and integer
    weights, each row divided by its (exact) sum."""
    keys = _rmat_keys(own, n, d)
    keys = torch.unique(torch.cat([keys, torch.arange(n, device=DEV) * (n + 1)]))
    w = torch.randint(1, 1000, (keys.numel(),), generator=own, device=DEV)
    names = _shuffle(gen, n)
    keys, order = torch.sort(_relabelled(keys, n, names, names))
    w, rows = w[order], keys // n
    sums = torch.zeros(n, dtype=torch.int64, device=DEV).index_add_(0, rows, w)
    return _csr(n, n, keys, index, w.double() / sums[rows].double())


def _predictor(gen):
    """A row-size predictor trained on exact row counts of small products."""
    train = []
    for n, d, kind in ((4096, 16, "rmat"), (16384, 12, "rmat"), (8192, 8, "er"), (8192, 16, "er")):
        names = _shuffle(gen, n)
        A = _matrix(gen, gen, {"graph": kind, "n": n, "d": d, "value": "f64", "index": "i32"},
                    names, names)
        train.append((A, A))
    X, T = sg.sizer_training_set(train)
    params = sg.sizer_init(seed=7)
    sg.sizer_train(X, T, params, steps=400, batch=4096, lr=3e-3, seed=8)
    return params


def _stencil(gen, nx, ny, nz):
    """7-point stencil: random negative couplings, a dominant diagonal."""
    n = nx * ny * nz
    idx = torch.arange(n, device=DEV)
    x, y, z = idx % nx, (idx // nx) % ny, idx // (nx * ny)
    keys = [idx * n + idx]
    for coord, size, stride in ((x, nx, 1), (y, ny, nx), (z, nz, nx * ny)):
        for sign in (-1, 1):
            ok = (coord + sign >= 0) & (coord + sign < size)
            keys.append(idx[ok] * n + idx[ok] + sign * stride)
    keys = torch.sort(torch.cat(keys)).values
    val = -0.5 - torch.rand(keys.numel(), generator=gen, device=DEV, dtype=torch.float64)
    val[keys // n == keys % n] += 10.0
    return _csr(n, n, keys, "i32", val)


def _aggregation(nx, ny, nz):
    """One 1.0 per fine point: the coarse point of its 2 x 2 x 2 cell."""
    cx, cy, cz = (nx + 1) // 2, (ny + 1) // 2, (nz + 1) // 2
    n = nx * ny * nz
    idx = torch.arange(n, device=DEV)
    agg = (idx % nx) // 2 + cx * (((idx // nx) % ny) // 2 + cy * ((idx // (nx * ny)) // 2))
    R = sg.DeviceCSR(n, cx * cy * cz, torch.arange(n + 1, device=DEV), agg.to(torch.int32),
                     torch.ones(n, dtype=torch.float64, device=DEV))
    return R, (cx, cy, cz)


def _hierarchy(gen, case):
    dims = (case["nx"], case["ny"], case["nz"])
    A = _stencil(gen, *dims)
    Rs = []
    for _ in range(case["levels"]):
        R, dims = _aggregation(*dims)
        Rs.append(R)
    return A, Rs


def _batch(own, gen, case):
    r = np.random.default_rng(case["count"] * 1000003 + case["nmax"])
    ns = np.floor(np.exp(r.uniform(math.log(case["nmin"]), math.log(case["nmax"]),
                                   case["count"]))).astype(int)
    ds = r.integers(case["dmin"], case["dmax"] + 1, case["count"])
    pairs = []
    for n, d in zip(ns, ds):
        one = {"graph": "er", "n": int(n), "d": int(d), "value": case["value"],
               "index": case["index"]}
        rows, inner, cols = (_shuffle(gen, int(n)) for _ in range(3))
        pairs.append((_matrix(own, gen, one, rows, inner), _matrix(own, gen, one, inner, cols)))
    return pairs


def _inputs(case, seed):
    gen, own = _generator(seed), _own_generator(case)
    op = case["op"]
    if op == "galerkin":
        return _hierarchy(gen, case)
    if op == "batch":
        return _batch(own, gen, case)
    if op == "mcl":
        return _markov(own, gen, case["n"], case["d"], case["index"]), gen
    names = _shuffle(gen, case["n"])
    if op == "merge":
        return [_matrix(own, gen, case, names, names) for _ in range(case["c"])]
    return _matrix(own, gen, case, names, names)


# -------------------------------------------------------------------- run
def prepare(case, seed):
    op = case["op"]
    state = {"case": case, "in": _inputs(case, seed)}
    if op == "mcl":
        M, gen = state["in"]
        state["in"], state["params"] = M, _predictor(gen)
    elif op == "batch":
        state["in"] = ([a for a, _ in state["in"]], [b for _, b in state["in"]])
    elif op == "galerkin":
        A, Rs = state["in"]
        chain = amg.GalerkinChain(A, Rs, torch.cuda.Stream(), persistent=case["persistent"])
        torch.cuda.synchronize()
        chain.run_eager()
        torch.cuda.synchronize()
        chain.check()
        chain.capture()
        # the operators' sizes depend on the grid alone: the arrays are viewed once
        state["chain"] = chain
        state["out"] = _chain_outputs(chain)
    torch.cuda.synchronize()
    return state


def _chain_outputs(chain):
    return [_arrays(M) for M in chain.intermediates() + chain.results()]


def _arrays(C):
    return {"rowptr": C.rowptr, "col": C.col, "val": C.val}


def run(state):
    case, X = state["case"], state["in"]
    op = case["op"]
    if op == "spgemm":
        return _arrays(sg.spgemm(X, X, semiring=_semiring(case)))
    if op == "masked":
        return _arrays(sg.masked_spgemm(X, X, X))
    if op == "kslice":
        return _arrays(sg.spgemm_kslice(X, X, case["c"])[0])
    if op == "merge":
        return _arrays(sg.merge(X, semiring=_semiring(case)))
    if op == "batch":
        p = sg.batch_plan(X[0], X[1], semiring=_semiring(case))
        rowptr, nnz = sg.symbolic(p)
        col, val = sg.alloc_output(p, nnz)
        sg.numeric(p, rowptr, col, val)
        p.close()
        return {"rowptr": rowptr, "col": col, "val": val}
    if op == "galerkin":
        state["chain"].replay()
        return state["out"]
    if op == "mcl":
        return _arrays(sg.mcl_step(X, THRESHOLD, state["params"], MARGIN))
    return _arrays(sg.transpose(X))


def _semiring(case):
    return sg.OR_AND if case["value"] == "none" else sg.PLUS_TIMES


# ------------------------------------------------------------------- work
def _bytes(*arrays):
    return float(sum(t.numel() * t.element_size() for t in arrays if t is not None))


def _matrix_bytes(M):
    return _bytes(M.rowptr, M.col, M.val)


def _products(A, B):
    lens = B.rowptr[1:] - B.rowptr[:-1]
    return float(lens[A.col.long()].sum())


def work(case):
    """Counted on the inputs of seed 0: every input and every output once, two
    operations per scalar product and one per merged entry."""
    state = prepare(case, 0)
    X, op = state["in"], case["op"]
    out = run(state)
    torch.cuda.synchronize()
    outs = out if isinstance(out, list) else [out]
    written = sum(_bytes(o["rowptr"], o["col"], o["val"]) for o in outs)
    if op == "merge":
        read, flops = sum(map(_matrix_bytes, X)), float(sum(M.nnz for M in X))
    elif op == "batch":
        read = sum(map(_matrix_bytes, X[0] + X[1]))
        flops = 2 * sum(_products(a, b) for a, b in zip(*X))
    elif op == "galerkin":
        A, Rs = X
        T, coarse = state["chain"].intermediates(), state["chain"].results()
        read = _matrix_bytes(A) + sum(map(_matrix_bytes, Rs))
        flops = 2 * float(sum(M.nnz for M in [A] + coarse[:-1]) + sum(M.nnz for M in T))
    else:
        read = _matrix_bytes(X)
        flops = 0.0 if op == "transpose" else 2 * _products(X, X)
    return {"bytes": read + written, "flops": flops}


# -------------------------------------------------------------- tolerance
def tolerance(case):
    """Products are rounded one by one and added in ascending inner index
    (partial products in ascending slice), which fixes every bit; the
    library states that order for all of its paths.  The order of a row sum in
    the clustering step is free: it was measured 1.9e-16 (2-norm) from the
    64-bit sums of another order, and four times that is allowed."""
    if case["op"] == "mcl":
        return {"rel": 8e-16}
    return "exact"


# ------------------------------------------------------------------ exact
STEP = 1 << 27  # products expanded at a time


def _wide(val):
    return None if val is None else val if val.dtype == torch.int64 else val.double()


def _reduce(keys, vals):
    """Distinct ascending keys and the sums of their values."""
    keys, order = torch.sort(keys)
    uniq, inverse = torch.unique_consecutive(keys, return_inverse=True)
    if vals is None:
        return uniq, None
    sums = torch.zeros(uniq.numel(), dtype=vals.dtype, device=DEV)
    return uniq, sums.index_add_(0, inverse, vals[order])


def _product(A, B, finish=None):
    """A.B in 64 bits by expansion, sorting and summing, in blocks of rows;
    finish(row numbers, columns, values) filters a block of whole rows."""
    lens = (B.rowptr[1:] - B.rowptr[:-1])[A.col.long()]
    before = torch.zeros(A.nnz + 1, dtype=torch.int64, device=DEV)
    before[1:] = lens.cumsum(0)
    ends = before[A.rowptr].cpu().numpy()
    rows_of = torch.repeat_interleave(torch.arange(A.nrows, device=DEV),
                                      A.rowptr[1:] - A.rowptr[:-1])
    va, vb = _wide(A.val), _wide(B.val)
    got_rows, got_cols, got_vals = [], [], []
    r0 = 0
    while r0 < A.nrows:
        r1 = max(r0 + 1, int(np.searchsorted(ends, ends[r0] + STEP, side="right")) - 1)
        p0, p1 = int(A.rowptr[r0]), int(A.rowptr[r1])
        n = lens[p0:p1]
        entry = torch.repeat_interleave(torch.arange(p0, p1, device=DEV), n)
        at = torch.arange(entry.numel(), device=DEV) - (before[entry] - before[p0])
        q = B.rowptr[A.col.long()[entry]] + at
        keys = rows_of[entry] * B.ncols + B.col.long()[q]
        vals = None if va is None else va[entry] * vb[q]
        keys, vals = _reduce(keys, vals)
        rows, cols = keys // B.ncols, keys % B.ncols
        if finish is not None:
            rows, cols, vals = finish(rows, cols, vals)
        got_rows.append(torch.bincount(rows - r0, minlength=r1 - r0))
        got_cols.append(cols.to(A.col.dtype))
        got_vals.append(vals)
        r0 = r1
    rowptr = torch.zeros(A.nrows + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cat(got_rows).cumsum(0)
    return sg.DeviceCSR(A.nrows, B.ncols, rowptr, torch.cat(got_cols),
                        None if va is None else torch.cat(got_vals))


def _transposed(A):
    rows = torch.repeat_interleave(torch.arange(A.nrows, device=DEV), A.rowptr[1:] - A.rowptr[:-1])
    keys, order = torch.sort(A.col.long() * A.nrows + rows)
    rowptr = torch.zeros(A.ncols + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.bincount(A.col.long(), minlength=A.ncols).cumsum(0)
    return sg.DeviceCSR(A.ncols, A.nrows, rowptr, (keys % A.nrows).to(A.col.dtype),
                        None if A.val is None else _wide(A.val)[order])


def _pruned(n):
    def finish(rows, cols, vals):
        keep = vals >= THRESHOLD
        rows, cols, vals = rows[keep], cols[keep], vals[keep]
        sums = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, rows, vals)
        return rows, cols, vals / sums[rows]
    return finish


def _inside(M):
    pattern = torch.repeat_interleave(torch.arange(M.nrows, device=DEV),
                                      M.rowptr[1:] - M.rowptr[:-1]) * M.ncols + M.col.long()

    def finish(rows, cols, vals):
        keys = rows * M.ncols + cols
        at = torch.searchsorted(pattern, keys).clamp_(max=pattern.numel() - 1)
        keep = pattern[at] == keys
        return rows[keep], cols[keep], vals[keep]
    return finish


def _concatenated(Cs):
    parts = [Cs[0].rowptr[:1]]
    base = 0
    for C in Cs:
        parts.append(C.rowptr[1:] + base)
        base += C.nnz
    return {"rowptr": torch.cat(parts), "col": torch.cat([C.col for C in Cs]),
            "val": None if Cs[0].val is None else torch.cat([C.val for C in Cs])}


def exact(case, seed):
    """What run() returns, by expansion and sorting in 64 bits on plain torch."""
    op, X = case["op"], _inputs(case, seed)
    if op == "masked":
        return _arrays(_product(X, X, _inside(X)))
    if op == "merge":
        n = X[0].ncols
        keys = torch.cat([torch.repeat_interleave(torch.arange(n, device=DEV),
                                                  M.rowptr[1:] - M.rowptr[:-1]) * n + M.col.long()
                          for M in X])
        keys, vals = _reduce(keys, None if X[0].val is None else torch.cat([_wide(M.val) for M in X]))
        return _arrays(_csr(n, n, keys, case["index"], vals))
    if op == "batch":
        return _concatenated([_product(a, b) for a, b in X])
    if op == "galerkin":
        A, Rs = X
        T, coarse = [], []
        for R in Rs:
            T.append(_product(_transposed(R), A))
            A = _product(T[-1], R)
            coarse.append(A)
        return [_arrays(M) for M in T + coarse]
    if op == "mcl":
        return _arrays(_product(X[0], X[0], _pruned(case["n"])))
    if op == "transpose":
        return _arrays(_transposed(X))
    return _arrays(_product(X, X))
