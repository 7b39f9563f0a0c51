"""GPU parity: the CUDA library (through the C ABI) against the CPU oracle,
element by element, on seeded inputs that span every row class (empty, the
four hash bins, dense rows with several column chunks), ragged tails, both
index types and every value type."""
import numpy as np
import pytest

import oracle
from paper_1510_00844_gb300 import inputs
from tests.parity import assert_pattern_equal, assert_values_close, rows_subset

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import torch
    assert torch.cuda.is_available()
    from paper_1510_00844_gb300 import spgemm
    return spgemm


def run(sg, A, B, semiring=0, checked=True):
    dA, dB = sg.to_device(A), sg.to_device(B)
    return sg.spgemm(dA, dB, semiring=semiring, checked=checked, verify=True)


SEMIRING = {0: "plus_times", 1: "or_and", 2: "min_plus", 3: "min_select2nd"}

# value type, semiring and index type of the row-size tests
VALUE_FORMS = [("u01_f64", 0, np.int32), ("int", 0, np.int32), ("none", 1, np.int32),
               ("u01_f64", 0, np.int64), ("none", 1, np.int64), ("u01_f64", 2, np.int32),
               ("int", 2, np.int64), ("u01_f64", 3, np.int64), ("int", 3, np.int32)]


def check_product(sg, A, B, dtype="f64"):
    C = run(sg, A, B)
    R = oracle.spgemm(A, B)
    assert_pattern_equal(C, R)
    assert_values_close(C, R, A, B, dtype)
    return C, R


def test_er_config_small(sg):
    # Erdos-Renyi, n = 16384, exactly 8 distinct rows per column, int32, f64
    A = inputs.er_column_regular(16384, 8, inputs.BASE_SEED + 1)
    C, R = check_product(sg, A, A)
    # same k order and no fused multiply-add: bit-exact in practice
    assert np.array_equal(C.to_host()[2], R.val)


@pytest.mark.parametrize("shape", [(1, 1, 1), (7, 1, 9), (1, 40, 1), (33, 65, 31), (300, 200, 500)])
@pytest.mark.parametrize("density", [0.0, 0.03, 0.3])
def test_random_shapes(sg, shape, density):
    m, l, n = shape
    A = inputs.random_csr(m, l, density, 11 + m, empty_rows=0.2)
    B = inputs.random_csr(l, n, density, 12 + n, empty_rows=0.2)
    check_product(sg, A, B)


@pytest.mark.parametrize("scale", [10, 12, 14])
def test_rmat_dense_rows(sg, scale):
    A = inputs.rmat(scale)
    C, R = check_product(sg, A, A)
    assert np.array_equal(C.to_host()[2], R.val)


def test_rmat_int64_indices(sg):
    A = inputs.rmat(12, index_dtype=np.int64)
    check_product(sg, A, A)


@pytest.mark.parametrize("value", ["int", "u11_f32"])
def test_value_types(sg, value):
    A = inputs.rmat(12, value=value)
    dtype = {"int": "i64", "u11_f32": "f32"}[value]
    C = run(sg, A, A)
    R = oracle.spgemm(A, A)
    assert_pattern_equal(C, R)
    assert_values_close(C, R, A, A, dtype)


def test_boolean_semiring(sg):
    A = inputs.rmat(12)
    Cb = run(sg, A.pattern(), A.pattern(), semiring=1)
    assert Cb.val is None
    R = oracle.spgemm(A.pattern(), A.pattern(), semiring="or_and")
    assert_pattern_equal(Cb, R)
    # OR_AND on valued inputs ignores values
    Cv = run(sg, A, A, semiring=1)
    assert_pattern_equal(Cv, R)


def bin_edge_case():
    """A with rows whose flops sit on every class edge: 0, 1, 32, 33, 128,
    129, 512, 513, 1024, 1025, 4096, plus one row hitting every B row.  B has
    rows of length 1..64 and two long rows (3000 and 20000 columns)."""
    rng = np.random.default_rng(5)
    n = 40000
    lensB = np.concatenate([np.arange(1, 65), [3000, 20000]])
    rowsB, colsB = [], []
    for k, L in enumerate(lensB):
        c = np.sort(rng.choice(n, size=L, replace=False))
        rowsB.append(np.full(L, k))
        colsB.append(c)
    B = inputs.coo_to_csr(len(lensB), n, np.concatenate(rowsB), np.concatenate(colsB),
                          rng.random(int(lensB.sum())), np.int32, sum_duplicates=False)
    targets = [0, 1, 32, 33, 128, 129, 512, 513, 1024, 1025, 4096]
    rowsA, colsA = [], []
    for i, t in enumerate(targets):
        # greedy subset of B rows (distinct k) summing to t
        rem, ks = t, []
        for k in np.argsort(-lensB):
            if lensB[k] <= rem and k not in ks and lensB[k] < 20000:
                ks.append(k)
                rem -= lensB[k]
        assert rem == 0
        rowsA += [i] * len(ks)
        colsA += list(ks)
    i = len(targets)
    rowsA += [i] * len(lensB)
    colsA += list(range(len(lensB)))
    A = inputs.coo_to_csr(i + 1, len(lensB), np.array(rowsA), np.array(colsA),
                          rng.random(len(rowsA)), np.int32, sum_duplicates=False)
    return A, B, targets


def test_class_edges_and_long_rows(sg):
    A, B, targets = bin_edge_case()
    fl = oracle.row_flops(A, B)
    assert list(fl[:len(targets)]) == targets
    C, R = check_product(sg, A, B)
    assert np.array_equal(C.to_host()[2], R.val)


def test_single_huge_row(sg):
    # one row selecting every row of an R-MAT matrix: dense accumulator over
    # all chunks, streaming of long B rows
    B = inputs.rmat(13)
    A = inputs.CSR(1, B.nrows, np.array([0, B.nrows]), np.arange(B.nrows, dtype=np.int32),
                   np.random.default_rng(1).random(B.nrows))
    check_product(sg, A, B)


def test_hypersparse_int64_columns(sg):
    # n > 2^31 columns, few entries: int64 indices end to end (hash rows only)
    rng = np.random.default_rng(3)
    n = (1 << 33) + 7
    m, l = 50, 60
    rA = rng.integers(0, m, 200)
    cA = rng.integers(0, l, 200)
    A = inputs.coo_to_csr(m, l, rA, cA, rng.random(200), np.int64)
    rB = rng.integers(0, l, 300)
    cB = rng.integers(0, n, 300)
    B = inputs.coo_to_csr(l, n, rB, cB, rng.random(300), np.int64)
    C = run(sg, A, B)
    # the oracle's dense accumulator is O(n): relabel B's distinct columns
    # 0..u-1 (monotone, so every row stays sorted), multiply, map back
    uniq = np.unique(B.col)
    Bc = inputs.CSR(l, len(uniq), B.rowptr, np.searchsorted(uniq, B.col), B.val)
    Rc = oracle.spgemm(A, Bc)
    R = oracle.OCSR(Rc.nrows, n, Rc.rowptr, uniq[Rc.col], Rc.val)
    assert_pattern_equal(C, R)
    assert_values_close(C, R)
    assert C.col.dtype.itemsize == 8 and int(C.col.max()) > 2**31


def test_empty_operands(sg):
    A = inputs.CSR(5, 4, np.zeros(6, dtype=np.int64), np.zeros(0, dtype=np.int32), np.zeros(0))
    B = inputs.random_csr(4, 7, 0.5, 1, index_dtype=np.int32)
    C = run(sg, A, B)
    assert C.nnz == 0 and np.array_equal(C.to_host()[0], np.zeros(6))
    Z = inputs.CSR(0, 4, np.zeros(1, dtype=np.int64), np.zeros(0, dtype=np.int32), np.zeros(0))
    C = run(sg, Z, B)
    assert C.nnz == 0 and C.nrows == 0


def test_determinism_bitwise(sg):
    A = inputs.rmat(13)
    dA = sg.to_device(A)
    C1 = sg.spgemm(dA, dA)
    C2 = sg.spgemm(dA, dA)
    assert bool((C1.val == C2.val).all()) and bool((C1.col == C2.col).all())


def test_checked_mode_rejects_invalid_csr(sg):
    A = inputs.random_csr(10, 10, 0.3, 2, index_dtype=np.int32)
    bad = A.col.copy()
    r = int(np.argmax(np.diff(A.rowptr) >= 2))
    bad[A.rowptr[r]], bad[A.rowptr[r] + 1] = bad[A.rowptr[r] + 1], bad[A.rowptr[r]]
    Abad = inputs.CSR(10, 10, A.rowptr, bad, A.val)
    with pytest.raises(sg.SpgemmError) as ei:
        run(sg, Abad, A, checked=True)
    assert ei.value.status == 2
    oob = A.col.copy()
    oob[-1] = 10
    with pytest.raises(sg.SpgemmError) as ei:
        run(sg, inputs.CSR(10, 10, A.rowptr, oob, A.val), A, checked=True)
    assert ei.value.status == 2


@pytest.mark.parametrize("c", [1, 2, 3, 4, 8, 16])
def test_kslice_merge(sg, c):
    A = inputs.rmat(12)
    dA = sg.to_device(A)
    C, parts = sg.spgemm_kslice(dA, dA, c, verify=True)
    ref_parts = [oracle.spgemm(As, Bs) for As, Bs in oracle.kslice(A, A, c)]
    for P, R in zip(parts, ref_parts):
        assert_pattern_equal(P, R)
        assert np.array_equal(P.to_host()[2], R.val)
    S = oracle.sum_partials(ref_parts)
    assert_pattern_equal(C, S)
    assert np.array_equal(C.to_host()[2], S.val)     # same order as the definition
    U = oracle.spgemm(A, A)
    assert_pattern_equal(C, U)
    assert_values_close(C, U, A, A)


def test_kslice_bounds_match_oracle(sg):
    A = inputs.rmat(11)
    dA = sg.to_device(A)
    for c in (1, 3, 4, 7):
        b = sg.kslice_bounds(dA, c).cpu().numpy()
        for s, (As, _) in enumerate(oracle.kslice(A, A, c)):
            assert np.array_equal(b[s + 1] - b[s], np.diff(As.rowptr))


def test_merge_integer_and_bool(sg):
    A = inputs.rmat(11, value="int")
    dA = sg.to_device(A)
    C, _ = sg.spgemm_kslice(dA, dA, 4, verify=True)
    R = oracle.spgemm(A, A)
    assert_pattern_equal(C, R)
    assert np.array_equal(C.to_host()[2], R.val)
    Cb, _ = sg.spgemm_kslice(sg.to_device(A.pattern()), sg.to_device(A.pattern()), 3,
                             semiring=1, verify=True)
    assert_pattern_equal(Cb, R)


def test_merge_unaligned_column_arrays(sg):
    """Partials whose int32 column arrays do not start on a 16-byte boundary
    are counted one column per lane (the four-column loads need aligned
    arrays); the merged product is still the oracle's sum of the partials."""
    import torch

    A = inputs.rmat(11)
    dA = sg.to_device(A)
    _, parts = sg.spgemm_kslice(dA, dA, 4, verify=True)
    shifted = []
    for P in parts:
        buf = torch.empty(P.col.numel() + 1, dtype=P.col.dtype, device=P.col.device)
        buf[1:] = P.col
        shifted.append(sg.DeviceCSR(P.nrows, P.ncols, P.rowptr, buf[1:], P.val))
    assert shifted[0].col.data_ptr() % 16 != 0
    C = sg.merge(shifted, verify=True)
    S = oracle.sum_partials([oracle.spgemm(As, Bs) for As, Bs in oracle.kslice(A, A, 4)])
    assert_pattern_equal(C, S)
    assert np.array_equal(C.to_host()[2], S.val)


@pytest.mark.parametrize("c,value,idx", [(2, "u01_f64", np.int32), (3, "u01_f64", np.int32),
                                         (4, "u01_f64", np.int32), (4, "int", np.int64),
                                         (4, "none", np.int32)])
def test_staged_merge_matches_oracle(sg, c, value, idx):
    """The numeric merge with every list staged in shared memory by bulk
    asynchronous copies (spgemm_opts.merge_staged) gives the oracle's sum of
    the partials bit for bit, for rows spanning many windows (R-MAT 13) and
    lists whose arrays end off a 16-byte boundary."""
    import torch
    A = inputs.rmat(13, index_dtype=idx, value=value)
    dA = sg.to_device(A)
    semiring = 1 if value == "none" else 0
    _, parts = sg.spgemm_kslice(dA, dA, c, semiring=semiring, verify=True)
    ws = sg.merge_workspace(c, A.nrows, A.ncols, dA.rowptr.device)
    rp, nnz = sg.merge_symbolic(parts, ws, semiring)
    col = torch.empty(nnz, dtype=dA.col.dtype, device="cuda")
    val = None if value == "none" else torch.empty(nnz, dtype=dA.val.dtype, device="cuda")
    sg.merge_numeric(parts, ws, rp, col, val, semiring, staged=True)
    sg.merge_check(ws)
    C = sg.DeviceCSR(A.nrows, A.ncols, rp, col, val)
    ref = [oracle.spgemm(As, Bs, semiring="or_and" if value == "none" else "plus_times")
           for As, Bs in oracle.kslice(A, A, c)]
    S = oracle.sum_partials(ref, semiring="or_and" if value == "none" else "plus_times")
    assert_pattern_equal(C, S)
    if val is not None:
        assert np.array_equal(C.to_host()[2], S.val)


def test_rmat_scale18_sampled_rows(sg):
    """The full R-MAT scale-18 squaring in the benchmark's launch
    configuration; a seeded sample of rows (including the largest-flops rows)
    is recomputed by the oracle row by row."""
    A = inputs.rmat(18)
    dA = sg.to_device(A)
    C = sg.spgemm(dA, dA, verify=True)
    fl = oracle.row_flops(A, A)
    rng = np.random.default_rng(7)
    rows = np.unique(np.concatenate([np.argsort(-fl)[:8], rng.choice(A.nrows, 400, replace=False)]))
    R = oracle.spgemm(rows_subset(A, rows), A)
    rp = C.rowptr.cpu().numpy()
    col = C.col.cpu().numpy()
    val = C.val.cpu().numpy()
    for t, i in enumerate(rows):
        a, b = rp[i], rp[i + 1]
        ra, rb = R.rowptr[t], R.rowptr[t + 1]
        assert b - a == rb - ra
        assert np.array_equal(col[a:b], R.col[ra:rb])
        assert np.array_equal(val[a:b], R.val[ra:rb])
    # global invariants at full size
    assert int(rp[-1]) <= int(fl.sum())
    assert np.all(np.diff(rp) <= np.minimum(fl, A.ncols))


@pytest.mark.parametrize("c", [1, 4, 16])
def test_hypersparse_kslices(sg, c):
    """k-slices multiplied as DCSR views of their nonempty rows (many rows of
    a slice are empty) give the same partials and the same merged product as
    the plain slices; row panels too."""
    A = inputs.rmat(12, seed=101)
    dA = sg.to_device(A)
    C1, P1 = sg.spgemm_kslice(dA, dA, c)
    C2, P2 = sg.spgemm_kslice(dA, dA, c, hypersparse=True)
    for a, b in zip(P1, P2):
        assert bool((a.rowptr == b.rowptr).all()) and bool((a.col == b.col).all())
        assert bool((a.val == b.val).all())
    assert bool((C1.rowptr == C2.rowptr).all()) and bool((C1.col == C2.col).all())
    assert bool((C1.val == C2.val).all())
    ids, v = sg.dcsr_view(dA)
    empty = np.diff(A.rowptr) == 0
    assert v.nrows == int((~empty).sum())
    assert np.array_equal(ids.cpu().numpy(), np.flatnonzero(~empty))
    R = oracle.spgemm(A, A)
    E = sg.dcsr_expand(sg.spgemm(v, dA), ids, A.nrows)
    assert_pattern_equal(E, R)
    assert np.array_equal(E.to_host()[2], R.val)


@pytest.mark.parametrize("idt", [np.int32, np.int64])
def test_short_rows_over_many_a_entries(sg, idt):
    """Rows of at most 32 products whose A entries are many, most of them
    pointing at empty rows of B (the table-free short-row path gathers their
    products over several batches of 32 A entries), rows of exactly 32
    products, and rows whose 32 products all land in one column."""
    rng = np.random.default_rng(41)
    n = 300
    # B rows 0..199 empty; 200..299 one entry in column 5; 300..399 one to
    # three entries in random columns
    rB, cB = [], []
    for k in range(200, 300):
        rB.append(k)
        cB.append(5)
    blen_r = rng.integers(1, 4, 100)
    for k, c in zip(range(300, 400), blen_r):
        cols = rng.choice(n, int(c), replace=False)
        rB += [k] * len(cols)
        cB += list(cols)
    B = inputs.coo_to_csr(400, n, np.array(rB), np.array(cB), rng.random(len(rB)), idt)
    blen = np.diff(B.rowptr)
    rows_A, cols_A = [], []

    def add(i, ks):
        ks = sorted(set(int(k) for k in ks))
        rows_A.extend([i] * len(ks))
        cols_A.extend(ks)

    for i in range(64):
        empty = rng.choice(200, 70, replace=False)
        if i < 16:          # a few products among many empty rows
            add(i, list(empty) + list(rng.choice(np.arange(300, 400), 6, replace=False)))
        elif i < 32:        # exactly 32 products
            ks, left = [], 32
            for k in rng.permutation(np.arange(300, 400)):
                if blen[k] <= left:
                    ks.append(k)
                    left -= blen[k]
                if left == 0:
                    break
            ks += list(range(200, 200 + left))      # one product each
            add(i, list(empty) + ks)
        elif i < 48:        # 32 products, all in column 5
            add(i, list(empty) + list(rng.choice(np.arange(200, 300), 32, replace=False)))
        else:               # half in column 5, half anywhere
            ks = list(rng.choice(np.arange(200, 300), 12, replace=False))
            ks += list(rng.choice(np.arange(300, 400), 5, replace=False))
            add(i, list(empty) + ks)
    A = inputs.coo_to_csr(64, 400, np.array(rows_A), np.array(cols_A), rng.random(len(rows_A)), idt)
    fl = oracle.row_flops(A, B)
    assert fl.max() <= 32 and (fl == 32).sum() >= 32 and np.diff(A.rowptr).min() > 32
    C, R = check_product(sg, A, B)
    assert np.array_equal(C.to_host()[2], R.val)
    assert np.all(np.diff(R.rowptr)[32:48] == 1)
    # the same rows in slot mode (learned sizing with an untrained predictor:
    # slots too small are re-run exactly)
    dA, dB = sg.to_device(A), sg.to_device(B)
    L, _ = sg.learned_multiply(dA, dB, sg.sizer_init(seed=9), 0.0)
    Lc = sg.compact(L)
    assert np.array_equal(Lc.rowptr.cpu().numpy(), R.rowptr)
    assert np.array_equal(Lc.col.cpu().numpy().astype(np.int64), R.col)
    assert np.array_equal(Lc.val.cpu().numpy(), R.val)


@pytest.mark.parametrize("c", [1, 2, 4, 9, 32])
@pytest.mark.parametrize("value", ["u01_f64", "u11_f32", "int", "none"])
def test_merge_row_sizes(sg, c, value):
    """Row totals at the edges of a numeric chunk (512 entries), a count chunk
    (2048) and of the rows cut into segments (beyond 8192); columns that fill a
    chunk's span (16384), that leave gaps wider than it, and lists of very
    unequal length."""
    rng = np.random.default_rng(c)
    totals = [0, 1, 2, 31, 511, 512, 513, 2047, 2048, 2049, 8191, 8192, 8193, 20000]
    n = 200_000
    rows = [(t, span, skew) for t in totals for span in (0, 16384, n) for skew in (False, True)]
    parts = []
    for s in range(c):
        cols = []
        for t, span, skew in rows:
            k = t // c if not skew else (t - (c - 1) * (t // (8 * c)) if s == 0 else t // (8 * c))
            width = max(k, span if span else t)        # span 0: columns side by side
            pick = rng.choice(width, size=k, replace=False) if width else np.zeros(0, np.int64)
            cols.append(np.sort(pick) + (n - width if skew else 0))
        lens = [x.size for x in cols]
        col = np.concatenate(cols)
        rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
        parts.append(inputs.CSR(len(rows), n, rp, col.astype(np.int32 if c % 2 else np.int64),
                                inputs.draw_values(rng, col.size, value)))
    sr = 1 if value == "none" else 0
    C = sg.merge([sg.to_device(P) for P in parts], semiring=sr, verify=True)
    S = oracle.sum_partials([oracle.OCSR(P.nrows, P.ncols, P.rowptr, P.col.astype(np.int64),
                                         None if P.val is None else P.val.astype(
                                             np.float64 if value == "u11_f32" else P.val.dtype))
                             for P in parts])
    rp, col, val = C.to_host()
    assert np.array_equal(rp, S.rowptr) and np.array_equal(col.astype(np.int64), S.col)
    if value == "u11_f32":
        # c - 1 additions of float32, each rounded to at most u = 2^-24 of a sum below c
        assert np.all(np.abs(val - S.val) <= (c - 1) * c * 2.0 ** -24)
    elif val is not None:
        assert np.array_equal(val, S.val)


def test_merge_more_long_rows_than_listed(sg):
    """More rows of over 8192 entries than the list of long rows holds (4096):
    the others are merged whole.  Even and odd columns give every column."""
    import torch

    m, n = 4200, 8400
    cols = torch.arange(n, device="cuda", dtype=torch.int32)
    parts = []
    for s in (0, 1):
        rp = torch.arange(m + 1, device="cuda", dtype=torch.int64) * (n // 2)
        col = cols[s::2].repeat(m)
        parts.append(sg.DeviceCSR(m, n, rp, col, col.double()))
    C = sg.merge(parts, verify=True)
    assert bool((C.rowptr == torch.arange(m + 1, device="cuda") * n).all())
    assert bool((C.col.view(m, n) == cols).all())
    assert bool((C.val.view(m, n) == cols.double()).all())


@pytest.mark.parametrize("n", [900, (1 << 25) - 1, 1 << 25])
@pytest.mark.parametrize("value,sr,index", VALUE_FORMS)
def test_rows_of_33_to_128_products(sg, n, value, sr, index):
    """Rows around the bounds of the register sort (64 and 128 products) with
    all columns distinct, all equal and mixed, over many A entries and over
    few, the last column among them; n = 2^25 is the first width whose rows
    keep the table."""
    rng = np.random.default_rng(n % 1000 + len(value))
    lens = [0, 1, 2, 3, 31, 32, 33, 64, 65, 100]        # one row of B per length and style
    styles = ["spread", "left", "right"]
    cols = []
    for k in lens:
        for s in styles:
            c = rng.choice(min(n, 5000), k, replace=False) if s == "spread" else np.arange(k)
            cols.append(np.sort(c if s != "right" else n - k + c))
    rp = np.concatenate([[0], np.cumsum([c.size for c in cols])]).astype(np.int64)
    col = np.concatenate(cols).astype(index)
    B = inputs.CSR(len(cols), n, rp, col, inputs.draw_values(rng, col.size, value))
    size = np.diff(rp)
    rows = []
    for target in [33, 48, 63, 64, 65, 96, 127, 128, 129, 200]:
        for _ in range(6):
            pick, left = [], target
            for k in rng.permutation(len(cols)):
                if size[k] <= left:
                    pick.append(k)
                    left -= size[k]
            rows.append(np.sort(pick))
    rpA = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int64)
    colA = np.concatenate(rows).astype(index)
    A = inputs.CSR(len(rows), len(cols), rpA, colA, inputs.draw_values(rng, colA.size, value))
    C = run(sg, A, B, semiring=sr)
    R = oracle.spgemm(A, B, semiring=SEMIRING[sr])
    assert_pattern_equal(C, R)
    if value != "none":
        assert np.array_equal(C.to_host()[2], R.val)


@pytest.mark.parametrize("n,value,sr,index",
                         [(2000, "u01_f64", 0, np.int32), (16384, "none", 1, np.int32),
                          (16385, "u11_f32", 0, np.int32), (32768, "int", 0, np.int32),
                          (32769, "u01_f64", 0, np.int32), (262144, "u01_f64", 0, np.int32),
                          (262144, "none", 1, np.int32), (262145, "int", 0, np.int32)]
                         + [(n, *form) for n in (2000, 32768, 262144, 262145)
                            for form in VALUE_FORMS[3:]])
def test_rows_of_129_to_1024_products(sg, n, value, sr, index):
    """Rows at the edges of the bitmap-ranked bins, on both sides of the widths
    up to which they are ranked: all columns distinct, every column hit by many
    A entries, and single products over a thousand A entries between empty
    rows of B; the last column among them."""
    rng = np.random.default_rng(n % 1000 + len(value))
    lens = [0] * 40 + [1] * 1100 + [7, 31, 32, 33, 64, 100, 128, 129, 300, 512, 1024]
    cols = []
    for t, k in enumerate(lens):
        if t % 3 == 0:
            c = rng.choice(n, k, replace=False)
        elif t % 3 == 1:
            c = np.arange(k)
        else:
            c = n - k + np.arange(k)
        cols.append(np.sort(c))
    order = rng.permutation(len(lens))
    cols = [cols[t] for t in order]
    size = np.array([c.size for c in cols])
    B = inputs.CSR(len(cols), n, np.concatenate([[0], np.cumsum(size)]).astype(np.int64),
                   np.concatenate(cols).astype(index),
                   inputs.draw_values(rng, int(size.sum()), value))
    rows = []
    for target in [128, 129, 130, 511, 512, 513, 1000, 1023, 1024, 1025]:
        for single in (False, True):
            for _ in range(3):
                pick, left = [], target
                for k in rng.permutation(len(cols)):
                    if size[k] <= left and (not single or size[k] <= 1):
                        pick.append(k)
                        left -= size[k]
                    if left == 0:
                        break
                rows.append(np.sort(pick))
    colA = np.concatenate(rows).astype(index)
    rpA = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int64)
    A = inputs.CSR(len(rows), len(cols), rpA, colA, inputs.draw_values(rng, colA.size, value))
    C = run(sg, A, B, semiring=sr)
    R = oracle.spgemm(A, B, semiring=SEMIRING[sr])
    assert_pattern_equal(C, R)
    if value == "u11_f32":
        assert_values_close(C, R, A, B, "f32")
    elif value != "none":
        assert np.array_equal(C.to_host()[2], R.val)


@pytest.mark.parametrize("n,l,value,width", [(130, 300, "u01_f64", 128), (700, 200, "none", 128),
                                             (1025, 150, "u11_f32", 128), (2047, 120, "int", 128),
                                             (3001, 100, "u01_f64", 256),
                                             (16500, 60, "u01_f64", 1024)])
def test_dense_rows_in_narrow_chunks(sg, n, l, value, width):
    """Few columns, long rows: the chunks of the dense rows are narrowed (down to
    128 columns) so that a row makes several work units; 16500 columns keep
    the full width for float64.  Plain and learned sizing."""
    A = inputs.random_csr(90, l, 0.6, 31 + n, value=value, index_dtype=np.int32)
    B = inputs.random_csr(l, n, 0.5, 32 + n, value=value, index_dtype=np.int32, empty_rows=0.1)
    sr = 1 if value == "none" else 0
    info = sg.plan(sg.to_device(A), sg.to_device(B), semiring=sr).info()
    assert info["rows_dense"] > 0 and info["chunk_width"] == width
    C = run(sg, A, B, semiring=sr)
    R = oracle.spgemm(A, B, semiring="or_and" if sr else "plus_times")
    assert_pattern_equal(C, R)
    if value == "u11_f32":
        assert_values_close(C, R, A, B, "f32")
    elif value != "none":
        assert np.array_equal(C.to_host()[2], R.val)
    L, _ = sg.learned_multiply(sg.to_device(A), sg.to_device(B), sg.sizer_init(seed=3), 0.2,
                               semiring=sr)
    L = sg.compact(L) if L.rowend is not None else L
    assert bool((L.col == C.col).all()) and bool((L.rowptr == C.rowptr).all())
    if value != "none":
        assert bool((L.val == C.val).all())


@pytest.mark.parametrize("n,rows,l,density", [(40000, 40, 300, 0.2), (65600, 7, 40, 0.9),
                                              (200_000, 9, 30, 0.002), (1500, 60, 80, 0.99)])
@pytest.mark.parametrize("index", [np.int32, np.int64])
def test_pattern_of_dense_rows(sg, n, rows, l, density, index):
    """Dense rows of a pattern, from the bitmaps the symbolic pass keeps (all
    cases but the third, whose bitmaps would take more bytes than there are
    products) and, with a second numeric pass, from them again; nearly full and
    sparse words, widths that are not whole words or chunks."""
    rng = np.random.default_rng(n % 991)
    A = inputs.random_csr(rows, l, 0.9, 41 + l, value="none", index_dtype=index)
    cols = [np.flatnonzero(rng.random(n) < density) for _ in range(l)]
    cols[0] = np.array([0, n - 1])
    B = inputs.CSR(l, n, np.concatenate([[0], np.cumsum([c.size for c in cols])]).astype(np.int64),
                   np.concatenate(cols).astype(index), None)
    dA, dB = sg.to_device(A), sg.to_device(B)
    p = sg.plan(dA, dB, semiring=1)
    assert p.info()["rows_dense"] > 0
    rp, nnz = sg.symbolic(p)
    R = oracle.spgemm(A, B, semiring="or_and")
    for _ in range(2):
        col, val = sg.alloc_output(p, nnz)
        col.fill_(-1)
        sg.numeric(p, rp, col, val)
        sg.check(p)
        assert np.array_equal(rp.cpu().numpy(), R.rowptr)
        assert np.array_equal(col.cpu().numpy().astype(np.int64), R.col)


@pytest.mark.parametrize("value,sr,index", VALUE_FORMS + [("u11_f32", 0, np.int32)])
@pytest.mark.parametrize("n", [700, 2**23 - 1, 2**23])
def test_rows_of_129_to_512_products_sorted(sg, n, value, sr, index):
    """Rows on both sides of eight and sixteen keys per lane, with distinct
    columns, with columns that most B rows share and with the last column, on
    both sides of the width up to which a warp sorts them."""
    rng = np.random.default_rng(n % 1000 + len(value))
    lens = [0] * 8 + [1] * 300 + [3, 17, 32, 33, 63, 64, 100, 128] * 3
    cols = []
    for t, k in enumerate(lens):
        c = [rng.choice(n, k, replace=False), np.arange(k), n - k + np.arange(k)][t % 3]
        cols.append(np.sort(c))
    size = np.array([c.size for c in cols])
    B = inputs.CSR(len(cols), n, np.concatenate([[0], np.cumsum(size)]).astype(np.int64),
                   np.concatenate(cols).astype(index),
                   inputs.draw_values(rng, int(size.sum()), value))
    rows = []
    for target in [129, 160, 161, 255, 256, 257, 288, 289, 511, 512]:
        for most in (1, 40, 128):
            pick, left = [], target
            for k in rng.permutation(len(cols)):
                if size[k] <= min(left, most):
                    pick.append(k)
                    left -= size[k]
            rows.append(np.sort(pick))
    colA = np.concatenate(rows).astype(index)
    rpA = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int64)
    A = inputs.CSR(len(rows), len(cols), rpA, colA, inputs.draw_values(rng, colA.size, value))
    C = run(sg, A, B, semiring=sr)
    R = oracle.spgemm(A, B, semiring=SEMIRING[sr])
    assert_pattern_equal(C, R)
    if value == "u11_f32":
        assert_values_close(C, R, A, B, "f32")
    elif value != "none":
        assert np.array_equal(C.to_host()[2], R.val)


@pytest.mark.parametrize("c", [1, 2, 4])
@pytest.mark.parametrize("value", ["u01_f64", "none"])
@pytest.mark.parametrize("index", [np.int32, np.int64])
def test_merge_of_rows_that_do_not_ascend(sg, c, value, index):
    """A part with a row of one repeated column or of descending columns (short,
    and long enough to be cut into segments), which no chunk can take in
    order: counts and numeric pass end and report it.  Rows with a column below
    the chunk's first or after one beyond its span give a sum of some kind.
    Other rows of the same merge are not disturbed."""
    import torch

    n = 100_000
    sr = 1 if value == "none" else 0
    good = np.arange(0, n, 97)
    for bad, found in (([5] * 3000, True), (list(range(6000, 0, -1)), True),
                       (list(range(9000, 0, -1)) + [7] * 3000, True),
                       ([3, 40_000, 5], False), ([100] + [3] * 40 + list(range(200, 900)), False),
                       ([9, 2, 60_000, 1] * 200, False)):
        rng = np.random.default_rng(c)
        parts = []
        for s in range(c):
            rows = [good, np.array(bad if s == c - 1 else good), good]
            rp = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int64)
            col = np.concatenate(rows).astype(index)
            parts.append(sg.to_device(inputs.CSR(3, n, rp, col,
                                                 inputs.draw_values(rng, col.size, value))))
        ws = sg.merge_workspace(c, 3, n, "cuda")
        for count in (lambda: sg.merge_symbolic(parts, ws, sr),
                      lambda: sg.merge_symbolic_static(parts, sr)):
            try:
                count()
                assert not found
            except sg.SpgemmError as e:
                assert e.status == 2        # INVALID_CSR
        # the numeric pass with row pointers that leave room for every entry
        ws.zero_()
        room = good.size + len(bad)
        rp = torch.tensor([0, good.size, good.size + room, 2 * good.size + room], device="cuda")
        col = torch.zeros(int(rp[3]), dtype=parts[0].col.dtype, device="cuda")
        val = None if sr else torch.zeros(int(rp[3]), dtype=torch.float64, device="cuda")
        sg.merge_numeric(parts, ws, rp, col, val, sr)
        try:
            sg.merge_check(ws)
            assert not found
        except sg.SpgemmError as e:
            assert e.status in (2, 8)       # or the bad row's count differs
        col = col.cpu().numpy()
        assert np.array_equal(col[:good.size], good) and np.array_equal(col[-good.size:], good)
        if not sr:
            want = np.sum([p.val.cpu().numpy()[:good.size] for p in parts], axis=0)
            got = val.cpu().numpy()[:good.size]
            # c - 1 additions, each rounded to at most 2^-53 of a sum below c
            assert np.all(np.abs(got - want) <= c * c * 2.0 ** -53)


@pytest.mark.parametrize("n", [3000, 200_000, 1_800_000])
@pytest.mark.parametrize("index", [np.int32, np.int64])
def test_dense_rows_over_runs_of_every_kind(sg, n, index):
    """The run tables of B on rows at the edges of a warp's window (32 entries), of
    its step (128) and of the rows that several warps share (beyond 2048): runs
    of one or a few entries, one run over many windows, and both in turn; rows of
    A that are dense over them."""
    rng = np.random.default_rng(n % 997)
    lens = [0, 1, 2, 31, 32, 33, 64, 65, 127, 128, 129, 160, 161, 1023, 1024, 1025, 2047, 2048,
            2049, 2176, 2177, 2900, 5000, 20_000]
    cols = []
    for k in lens:
        if k > n:
            continue
        cols.append(rng.choice(n, k, replace=False))                       # spread
        cols.append(np.arange(k))                                          # side by side
        cols.append(n - k + np.arange(k))
        step = max(1, min(n // max(k, 1), 1500))
        cols.append(np.arange(k) * step)                                   # evenly
        half = np.concatenate([np.arange(k // 2), n - 1 - 40 * np.arange(k - k // 2)])
        cols.append(np.unique(np.clip(half, 0, n - 1)))                    # a block, then apart
    cols = [np.sort(c) for c in cols]
    size = np.array([c.size for c in cols])
    B = inputs.CSR(len(cols), n, np.concatenate([[0], np.cumsum(size)]).astype(np.int64),
                   np.concatenate(cols).astype(index), rng.random(int(size.sum())))
    rows = [np.sort(rng.choice(len(cols), k, replace=False)) for k in (1, 5, 20, 40, 60, 90)
            for _ in range(4)] + [np.arange(len(cols))]
    rows += [np.array([t]) for t in range(len(cols))]
    colA = np.concatenate(rows).astype(index)
    rpA = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int64)
    A = inputs.CSR(len(rows), len(cols), rpA, colA, rng.random(colA.size))
    C = run(sg, A, B)
    R = oracle.spgemm(A, B)
    assert_pattern_equal(C, R)
    assert np.array_equal(C.to_host()[2], R.val)


def test_pattern_with_row_pointers_of_another_product(sg):
    """Row pointers that are not the plan's: every row short and at the end of the
    arrays, in front of them, or beyond them.  Reported, and nothing is written
    outside the columns handed over."""
    import torch

    n, l = 40_000, 60
    A = inputs.random_csr(30, l, 0.9, 71, value="none", index_dtype=np.int32)
    B = inputs.random_csr(l, n, 0.05, 72, value="none", index_dtype=np.int32)
    p = sg.plan(sg.to_device(A), sg.to_device(B), semiring=1)
    assert p.info()["rows_dense"] == 30
    rp, nnz = sg.symbolic(p)
    room = torch.full((nnz + 2 * n,), -7, dtype=torch.int32, device="cuda")
    col = room[n:n + nnz]
    base = torch.arange(31, device="cuda")
    for other in (torch.full_like(rp, nnz), nnz - 30 + base, base - 15, rp + 1, rp.flip(0)):
        sg.numeric(p, other.to(torch.int64).contiguous(), col, None)
        with pytest.raises(sg.SpgemmError):
            sg.check(p)
        assert bool((room[:n] == -7).all()) and bool((room[n + nnz:] == -7).all())
        p = sg.plan(sg.to_device(A), sg.to_device(B), semiring=1)
        rp, nnz = sg.symbolic(p)
    sg.numeric(p, rp, col, None)
    sg.check(p)
    R = oracle.spgemm(A, B, semiring="or_and")
    assert np.array_equal(col.cpu().numpy().astype(np.int64), R.col)


def test_pattern_without_room_for_bitmaps(sg, monkeypatch):
    """A pattern plan takes any workspace from spgemm_workspace_least on, with the
    same result, and falls back to it where the device has no room for its
    bitmaps or, beside them, for C."""
    import torch

    n, l = 1_800_000, 30
    A = inputs.random_csr(60, l, 0.97, 81, value="none", index_dtype=np.int32)
    rng = np.random.default_rng(82)
    cols = [np.sort(rng.choice(n, 10_000, replace=False)) for _ in range(l)]
    B = inputs.CSR(l, n, (np.arange(l + 1) * 10_000).astype(np.int64),
                   np.concatenate(cols).astype(np.int32), None)
    dA, dB = sg.to_device(A), sg.to_device(B)
    R = oracle.spgemm(A, B, semiring="or_and")

    def right(rp, col):
        return (np.array_equal(rp.cpu().numpy(), R.rowptr)
                and np.array_equal(col.cpu().numpy().astype(np.int64), R.col))

    p = sg.plan(dA, dB, semiring=1)
    full, least = p.ws.numel(), p.least_workspace()
    assert p.info()["rows_dense"] == 60 and least < full
    for size in (full - 1, least, full, full + 1, least + 1):
        p.ws = sg._workspace(size, "cuda")
        rp, nnz = sg.symbolic(p)
        col, _ = sg.alloc_output(p, nnz)
        sg.numeric(p, rp, col, None)
        sg.check(p)
        assert p.ws.numel() == size and right(rp, col)
    p.ws = sg._workspace(least - 1, "cuda")
    with pytest.raises(sg.SpgemmError) as e:
        sg.symbolic(p)
    assert e.value.status == 4          # OUT_OF_MEMORY

    # no room for the larger workspace
    make, sizes = sg._workspace, []

    def small_only(nbytes, device):
        sizes.append(nbytes)
        if nbytes >= full:
            raise torch.OutOfMemoryError("no room")
        return make(nbytes, device)

    monkeypatch.setattr(sg, "_workspace", small_only)
    C = sg.spgemm(dA, dB, semiring=1, verify=True)
    assert full in sizes and sizes[-1] == least and right(C.rowptr, C.col)
    monkeypatch.setattr(sg, "_workspace", make)

    # no room for C beside it
    p = sg.plan(dA, dB, semiring=1)
    output = sg._output

    def beside_least(q, nnz):
        if q.ws.numel() > least:
            raise torch.OutOfMemoryError("no room")
        return output(q, nnz)

    monkeypatch.setattr(sg, "_output", beside_least)
    rp, nnz = sg.symbolic(p)
    col, _ = sg.alloc_output(p, nnz)
    sg.numeric(p, rp, col, None)
    sg.check(p)
    assert p.ws.numel() == least and right(rp, col)
