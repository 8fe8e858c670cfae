"""F3R's Arnoldi step over the sizes where its form changes: one and several
vectors per thread, 16 and 32 elements, and beyond what the registers of all
blocks hold. With n a multiple of four every step of an FP32 layer takes the
cooperative kernel; the same system with one decoupled unknown of zero more
(n + 1) has its basis vectors at unaligned distances, so three of four steps
take the separate kernels. The iterate after one outer step, far from
converged, must be the same."""
import numpy as np
import pytest

from paper_2604_13433_gb300 import inputs as I

from _gpu import P, dev, need_gpu

pytestmark = pytest.mark.gpu


def banded(n, extra):
    """Unit diagonal with -0.125 and -0.25 beside it and 1,000 away, and `extra` unknowns of their own."""
    i = np.arange(n, dtype=np.int64)
    offs = [(-1000, -0.25), (-1, -0.125), (0, 1.0), (1, -0.125), (1000, -0.25)]
    cols = np.stack([i + o for o, _ in offs], axis=1)
    ok = (cols >= 0) & (cols < n)
    vals = np.broadcast_to(np.array([v for _, v in offs]), cols.shape)
    rowptr = np.concatenate([[0], np.cumsum(ok.sum(axis=1))])
    rowptr = np.concatenate([rowptr, rowptr[-1] + 1 + np.arange(extra)])
    col = np.concatenate([cols[ok], n + np.arange(extra)]).astype(np.int32)
    val = np.concatenate([vals[ok], np.ones(extra)])
    return I.CSR(n + extra, n + extra, rowptr.astype(np.int64), col, val)


@pytest.mark.parametrize("n", [622592, 848160, 2490368, 2490372, 2744000, 4980736, 5088448])
def test_forms_of_the_arnoldi_step_agree(n):
    """Tolerance: the two forms differ in the FP32 sums of at most 33 products per
    thread, 33 x 2^-24 = 2e-6 of a sum each; six Arnoldi steps of a well-conditioned
    operator give at most about 1e-5 in x. A vector left out of a step changes x by
    its share of the vector, 1e-2 or more."""
    need_gpu()
    ps = P()
    b = I.uniform(n, seed=5, lo=-1.0, hi=1.0).astype(np.float64)
    out = []
    for extra in (0, 1):
        csr = banded(n, extra)
        A1 = ps.packsell_encode_csr(csr, fmt="sell_f64")
        A2 = ps.packsell_encode_csr(csr, fmt="sell_f32")
        A3 = ps.packsell_encode_csr(csr, fmt="fp16", D=15)
        x, info = ps.packsell_f3r(A1, A2, A3, dev(np.concatenate([b, np.zeros(extra)])), m1=4, m2=2, m3=2,
                                  m4=1, rtol=1e-14, max_iters=1, check=False)
        out.append((x.cpu().numpy(), info))
    (x, info), (y, info1) = out
    assert info["iters"] == info1["iters"] == 1 and 1e-6 < info["relres_true"] < 0.5
    assert abs(info["relres_true"] / info1["relres_true"] - 1) < 1e-4
    assert y[n] == 0.0
    err = np.linalg.norm(x - y[:n]) / np.linalg.norm(x)
    assert err < 1e-5, err
