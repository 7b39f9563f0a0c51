"""MCL epilogue on the GPU against the oracle, step by step: each GPU step's
input is the previous GPU output, the oracle prunes and renormalises the same
product.  Entries within 1e-12 (relative) of the threshold could fall on
either side of it; none may differ otherwise."""
import numpy as np
import pytest

import oracle
from paper_1510_00844_gb300 import inputs
from tests.parity import assert_pattern_equal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import torch
    assert torch.cuda.is_available()
    from paper_1510_00844_gb300 import spgemm
    return spgemm


@pytest.mark.parametrize("scale,steps,thr", [(10, 3, 1e-4), (10, 3, 1e-2), (14, 2, 1e-4)])
def test_mcl_steps_match_oracle(sg, scale, steps, thr):
    M = inputs.mcl_transition(scale)
    dM = sg.to_device(M)
    for step in range(steps):
        hostM = oracle.OCSR(M.nrows, M.ncols, *dM.to_host())
        C = sg.spgemm(dM, dM)
        R = oracle.mcl_prune_renorm(oracle.spgemm(hostM, hostM), thr)
        dM = sg.mcl_prune(C, thr)
        rp, col, val = dM.to_host()
        assert np.array_equal(rp, R.rowptr) and np.array_equal(col.astype(np.int64), R.col)
        np.testing.assert_allclose(val, R.val, rtol=1e-12)
        nz = np.diff(rp) > 0
        sums = np.add.reduceat(val, rp[:-1][nz]) if nz.any() else np.zeros(0)
        np.testing.assert_allclose(sums, 1.0, rtol=1e-12)


def test_mcl_on_slot_view_and_learned(sg):
    import torch
    M = inputs.mcl_transition(9)
    dM = sg.to_device(M)
    params = sg.sizer_init(seed=5)      # an untrained predictor: slots miss often
    A = sg.mcl_step(dM, 1e-3)
    B = sg.mcl_step(dM, 1e-3, params=params, margin=0.0)
    assert bool((A.rowptr == B.rowptr).all()) and bool((A.col == B.col).all())
    assert bool((A.val == B.val).all())


@pytest.mark.parametrize("thr", [0.25, 0.0, -0.5])
def test_prune_row_lengths_and_special_values(sg, thr):
    # rows at the edges of a warp's step (128 entries), of the rows a block
    # takes (beyond 2048) and of its step (1024); values around the threshold,
    # zeros of both signs, NaN and infinities
    rng = np.random.default_rng(5)
    lens = np.array([0, 1, 31, 32, 127, 128, 129, 2047, 2048, 2049, 3072, 3073, 7000, 0, 5])
    rowptr = np.concatenate([[0], np.cumsum(lens)])
    n = int(lens.max())
    col = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens]).astype(np.int32)
    val = rng.random(col.size) - 0.3
    val[rng.random(col.size) < 0.1] = 0.25
    val[rng.random(col.size) < 0.05] = np.nextafter(0.25, 0)
    val[rng.random(col.size) < 0.05] = -0.0
    special = slice(int(rowptr[6]), int(rowptr[7]))        # one row also holds NaN and infinities
    val[special][::7] = np.nan
    val[special][::11] = -np.inf
    val[special][::13] = np.inf
    C = inputs.CSR(lens.size, n, rowptr.astype(np.int64), col, val)
    P = sg.mcl_prune(sg.to_device(C), thr)
    rp, pc, pv = P.to_host()
    for i in range(lens.size):
        v, c = val[rowptr[i]:rowptr[i + 1]], col[rowptr[i]:rowptr[i + 1]]
        keep = v >= thr
        a, b = rp[i], rp[i + 1]
        assert b - a == keep.sum() and np.array_equal(pc[a:b], c[keep])
        with np.errstate(invalid="ignore"):
            s = v[keep].sum()
            want = v[keep] / s
        # a sum of k terms in any order is off by at most k u sum|v|, the
        # division by u
        # (an infinite sum leaves exact zeros)
        bound = 0.0
        if np.isfinite(s) and s != 0:
            bound = (keep.sum() + 2) * 2.0 ** -53 * np.abs(v[keep]).sum() / abs(s)
        ok = np.isfinite(want)
        assert np.array_equal(np.isnan(pv[a:b]), np.isnan(want))
        assert np.all(np.abs(pv[a:b][ok] - want[ok]) <= bound * np.abs(want[ok]))
