"""F3R's FP32 layers add their products in FP64 beyond what one thread holds, so
with at most one element per thread (n up to 155,648) the order of the unknowns
does not matter to them: a diagonal system and its permutation give permuted
solutions, up to the FP64 sums of the outer layer."""
import numpy as np
import pytest

from paper_2604_13433_gb300 import inputs as I

from _gpu import P, dev, need_gpu

pytestmark = pytest.mark.gpu


def diagonal(d):
    n = len(d)
    return I.CSR(n, n, np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), d)


@pytest.mark.parametrize("n", [1000, 40000, 40003, 155000])
def test_sums_do_not_depend_on_the_order(n):
    """Tolerance: FP64 sums of n terms differ by at most about n eps (3.4e-11 at
    155,000, and by its root, 1e-13, in practice); an FP32 sum of four products
    differs by 6e-8 of its size, which the few large entries of b do not average
    away."""
    need_gpu()
    ps = P()
    g = np.random.default_rng(n)
    d = (g.integers(512, 1536, n) / 1024.0).astype(np.float64)  # exact in binary16
    b = np.exp(3.0 * g.standard_normal(n))
    perm = g.permutation(n)

    def solve(d, b):
        csr = diagonal(d)
        A1 = ps.packsell_encode_csr(csr, fmt="sell_f64")
        A2 = ps.packsell_encode_csr(csr, fmt="sell_f32")
        A3 = ps.packsell_encode_csr(csr, fmt="fp16", D=15)
        x, info = ps.packsell_f3r(A1, A2, A3, dev(b), m2=4, m3=2, m4=1, rtol=1e-2)
        return x.cpu().numpy(), info

    x, info = solve(d, b)
    xp, infop = solve(d[perm], b[perm])
    assert info["iters"] == infop["iters"] == 1
    err = np.linalg.norm(x[perm] - xp) / np.linalg.norm(x)
    assert err < 1e-11, err
