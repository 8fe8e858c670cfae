"""SpMM with 32-byte X and Y rows (eight columns per lane, 256-bit loads) and the
layouts just beside it that take the other kernels: every column of Y has the
bits of the SpMV with that column of X."""
import numpy as np
import pytest

from paper_2604_13433_gb300 import inputs as I

from _gpu import P, dev, need_gpu, torch

pytestmark = pytest.mark.gpu


def _rows(n, width, seed):
    """Rows of 0 to `width` columns around the diagonal; the first has `width`."""
    rng = np.random.default_rng(seed)
    m = n + 2 * width
    rows = [np.sort(rng.choice(2 * width, size=width if i == 0 else rng.integers(0, width + 1),
                               replace=False)) + i for i in range(n)]
    rowptr = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int64)
    col = np.concatenate(rows).astype(np.int32)
    return I.CSR(n=n, m=m, rowptr=rowptr, col=col, val=rng.standard_normal(col.size).astype(np.float32))


CASES = {"stencil": I.stencil27((19, 11, 13), seed=5), "part_slice": _rows(31, 20, 1),
         "w8": _rows(1000, 8, 2), "w47": _rows(333, 47, 3), "w60": _rows(333, 60, 4)}


@pytest.mark.parametrize("fmt,D", [("fp16", 15), ("e8my", 3)])
@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("k", [4, 8, 16, 20, 24, 32, 40, 64, 72, 136])
def test_spmm_wide_rows(fmt, D, name, k):
    need_gpu()
    ps = P()
    csr = CASES[name]
    for sigma, explicit, pad, shift in ((1, False, 0, 0), (256, False, 8, 8), (64, True, 8, 0),
                                        (256, False, 8, 4), (256, False, 4, 0)):
        A = ps.packsell_encode_csr(csr, fmt=fmt, D=D, C=32, sigma=sigma, explicit_perm=explicit)
        X = torch.zeros((csr.m, k + pad), device="cuda")[:, shift:shift + k]
        X.copy_(dev(I.uniform(csr.m * k, seed=k).reshape(csr.m, k)))
        X[5, 3] = float("inf")  # only the rows that hold column 5 see it
        wide = torch.full((csr.n, k + 16), -7.0, device="cuda")
        Y = ps.packsell_spmm(A, X, wide[:, 8:8 + k])
        for q in {0, 3, k // 2, k - 1}:
            y = ps.packsell_spmv(A, X[:, q].contiguous())
            assert torch.equal(Y[:, q].contiguous().view(torch.int32), y.view(torch.int32))
        assert bool((wide[:, :8] == -7).all()) and bool((wide[:, 8 + k:] == -7).all())
