"""F3R where its vector kernels change form: vector lengths that are not a
multiple of four (the scalar tails and unaligned basis vectors), one thread's
worth of elements and less, Richardson counts of both parities and omega != 1,
and a matrix whose product has no Richardson epilogue."""
import numpy as np
import pytest

from paper_2604_13433_gb300 import inputs as I

from _gpu import P, dev, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(3, 3, 3), (16, 16, 16), (17, 13, 11), (30, 29, 41)])
@pytest.mark.parametrize("m4,omega", [(1, 1.0), (2, 1.0), (3, 1.0), (2, 0.9), (3, 0.9), (4, 0.9)])
def test_f3r_forms_agree(grid, m4, omega):
    """PackSELL and FP16 SELL run the same vector kernels and give the same
    iterates bit for bit; so does the PackSELL matrix pinned to variant 5, whose
    product has no epilogue; the solution meets the tolerance on the residual
    of the FP64 matrix."""
    need_gpu()
    ps = P()
    csr = I.diag_scaled(I.stencil27(grid, seed=3))
    b = I.uniform(csr.n, seed=5, lo=0.0, hi=1.0).astype(np.float64)
    A1 = ps.packsell_encode_csr(csr, fmt="sell_f64")
    A2 = ps.packsell_encode_csr(csr, fmt="sell_f32")
    xs = []
    for fmt, variant in (("fp16", 0), ("sell_f16", 0), ("fp16", 5)):
        A3 = ps.packsell_encode_csr(csr, fmt=fmt, D=15)
        if variant:
            ps.packsell_set_spmv_variant(A3, variant)
        x, info = ps.packsell_f3r(A1, A2, A3, dev(b), m4=m4, omega=omega, rtol=1e-9)
        assert info["relres_true"] < 1e-9
        xs.append(x.cpu().numpy())
    assert np.array_equal(xs[0], xs[1]) and np.array_equal(xs[0], xs[2])
    row = np.repeat(np.arange(csr.n), csr.row_lengths())
    r = b - np.bincount(row, weights=csr.val * xs[0][csr.col], minlength=csr.n)
    assert np.linalg.norm(r) < 1e-9 * np.linalg.norm(b) * (1 + 1e-6)
