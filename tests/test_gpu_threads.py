"""Host threads that call the library at once, each on its own stream, with sizes
that need different amounts of shared memory from the same kernels."""
import ctypes
import threading

import numpy as np
import pytest

import oracle
from paper_1510_00844_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import torch
    assert torch.cuda.is_available()
    from paper_1510_00844_gb300 import spgemm
    return spgemm


def in_threads(*work):
    """Each of `work` in a thread and a stream of its own, 2000 times; the first
    exception, if any, ends all."""
    import torch
    failed = []

    def loop(f):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(2000):
                    f()
                    if failed:
                        break
                torch.cuda.current_stream().synchronize()
        except Exception as e:      # noqa: BLE001  (handed to the main thread)
            failed.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=loop, args=(f,)) for f in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if failed:
        raise failed[0]


def wide(n, rows, l, nnz, seed):
    """rows x l times l x n, nnz entries in every row of B."""
    rng = np.random.default_rng(seed)
    A = inputs.random_csr(rows, l, 0.999, seed, index_dtype=np.int32)
    cols = [np.sort(rng.choice(n, nnz, replace=False)) for _ in range(l)]
    B = inputs.CSR(l, n, (np.arange(l + 1) * nnz).astype(np.int64),
                   np.concatenate(cols).astype(np.int32), rng.random(l * nnz))
    return A, B


@pytest.mark.parametrize("l,nnz,ns", [(20, 40, (190_000, 262_144)), (40, 60, (400_000, 1_500_000))])
def test_products_of_different_widths(sg, l, nnz, ns):
    # 800 products per row (ranked by a bitmap) and 2400 (dense)
    import torch
    made = []
    for n in ns:
        A, B = wide(n, 64, l, nnz, n % 1000)
        dA, dB = sg.to_device(A), sg.to_device(B)
        torch.cuda.synchronize()
        p = sg.plan(dA, dB, stream=torch.cuda.Stream())
        rp, nonzeros = sg.symbolic(p)
        made.append((p, rp, *sg.alloc_output(p, nonzeros), oracle.spgemm(A, B)))

    def product(t):
        p, rp, col, val, _ = made[t]

        def f():
            sg.symbolic(p, rp)
            sg.numeric(p, rp, col, val)
        return f

    in_threads(product(0), product(1))
    torch.cuda.synchronize()
    for p, rp, col, val, R in made:
        sg.check(p)
        assert np.array_equal(rp.cpu().numpy(), R.rowptr)
        assert np.array_equal(col.cpu().numpy().astype(np.int64), R.col)
        assert np.array_equal(val.cpu().numpy(), R.val)


def test_transposes_of_different_heights(sg):
    mats = [inputs.random_csr(4, m, 300.0 / m, m % 1000, index_dtype=np.int32)
            for m in (210_000, 450_000)]
    mats = [oracle.transpose(M) for M in mats]      # m x 4 with long columns
    mats = [inputs.CSR(M.nrows, M.ncols, M.rowptr, M.col.astype(np.int32), M.val) for M in mats]
    dev = [sg.to_device(M) for M in mats]
    got = [sg.transpose(M) for M in dev]
    made = []
    for M, T in zip(dev, got):
        c = sg._csr(M)
        ws = sg._workspace(sg._lib.spgemm_transpose_workspace_size(ctypes.byref(c)), "cuda")
        made.append((c, ws, [ctypes.c_void_p(x.zero_().data_ptr()) for x in (T.rowptr, T.col, T.val)]))

    def transposed(t):
        c, ws, out = made[t]

        def f():
            sg._check(sg._lib.spgemm_transpose(ctypes.byref(c), sg._stream(),
                                               ctypes.c_void_p(ws.data_ptr()), ws.numel(), *out))
        return f

    in_threads(transposed(0), transposed(1))
    for t, M in enumerate(mats):
        R = oracle.transpose(M)
        rp, col, val = got[t].to_host()
        assert np.array_equal(rp, R.rowptr) and np.array_equal(col.astype(np.int64), R.col)
        assert np.array_equal(val, R.val)
