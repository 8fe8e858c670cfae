"""Backward products in one pass over the words (dx = A^T dy, dval = dy_i x_j on
the pattern, each alone and both), in slices of 32 rows and in CSR order, at
the edges of their rounds and tiles."""
import numpy as np
import pytest

import oracle as O
from paper_2604_13433_gb300 import inputs as I

from _gpu import FMT, P, dev, need_gpu

pytestmark = pytest.mark.gpu


def _matrix(lengths, m, seed):
    """CSR with the given row lengths: ascending columns spread over [0, m)."""
    rng = np.random.default_rng(seed)
    rowptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    col = np.concatenate([np.sort(rng.choice(m, size=k, replace=False)) for k in lengths] or [[]])
    return I.CSR(n=len(lengths), m=m, rowptr=rowptr, col=col.astype(np.int32),
                 val=rng.standard_normal(rowptr[-1]).astype(np.float32))


# rows at the edges of a round of 16 words and of a tile of 253 words, empty
# rows, runs of one-word rows (a tile of 256 rows), long rows of several chunks
ROUNDS = [0, 1, 15, 16, 17, 31, 32, 33, 0, 48] * 7 + [5]
TILES = [0, 250, 1, 253, 254, 0, 255, 256, 257, 3, 700, 1] + [1] * 600 + [0] * 40 + [9, 1030, 2]


@pytest.mark.parametrize("fmt,D", [("fp16", 15), ("e8my", 4)])
@pytest.mark.parametrize("C,sigma,explicit,lengths", [
    (32, 1, False, ROUNDS), (32, 64, False, ROUNDS), (32, 64, True, ROUNDS), (32, 48, False, TILES),
    (32, 256, False, [3]), (1, 1, False, ROUNDS), (1, 1, False, TILES), (1, 64, False, TILES)])
def test_backward_one_pass(fmt, D, C, sigma, explicit, lengths):
    need_gpu()
    ps = P()
    m = 5000
    csr = _matrix(lengths, m, seed=len(lengths) + D)
    A = ps.packsell_encode_csr(csr, fmt=fmt, D=D, C=C, sigma=sigma, explicit_perm=explicit,
                               keep_rowptr=True)
    enc = O.encode(csr, C=C, sigma=sigma, D=D, fmt=FMT[fmt])
    row = np.repeat(np.arange(csr.n), csr.row_lengths())
    x, dy = I.uniform(m, seed=1), I.uniform(csr.n, seed=2)
    dy[::5] = 0.0
    # dx takes dy in the matrix's output order, dval in original order
    stored = ps.packsell_storage_rows(A).cpu().numpy() if explicit else np.arange(csr.n)
    dy_x = np.empty_like(dy)
    dy_x[stored] = dy
    ref = O.csr_spmv_t_f64(csr, enc.deq, dy_x.astype(np.float64))
    # FP32 products and sums in any order: gamma_(c_j + 1) sum_i |a_ij dy_i|
    u = 2.0 ** -24
    cnt = np.bincount(csr.col, minlength=m) + 1.0
    tol = cnt * u / (1 - cnt * u) * O.csr_spmv_t_f64(csr, np.abs(enc.deq), np.abs(dy_x).astype(np.float64))
    want = (dy[row] * x[csr.col]).astype(np.float32)
    for need_dx, need_dval in ((True, True), (True, False), (False, True)):
        dx, dval = ps.packsell_spmv_backward(A, dev(x), dev(dy), need_dx=need_dx, need_dval=need_dval)
        if need_dx:
            assert np.all(np.abs(dx.cpu().numpy() - ref) <= tol)
        if need_dval:
            assert np.array_equal(dval.cpu().numpy().view(np.uint32), want.view(np.uint32))
