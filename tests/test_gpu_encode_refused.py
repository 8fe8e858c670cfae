"""A matrix whose rows are refused in every block of the encoder's counting pass
(a left offset too small for Eq. 4): each block takes the error or leaves early
as a whole, and the next encode is that of a fresh library."""
import pytest

from paper_2604_13433_gb300 import inputs as I

from _gpu import P, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [32, 1])
def test_left_offset_refused_in_many_blocks(C):
    need_gpu()
    ps = P()
    csr = I.poisson5(700)
    want = ps.packsell_encode_csr(csr, fmt="fp16", C=C, sigma=1)
    for _ in range(3):
        with pytest.raises(ps.PackSELLError) as e:
            ps.packsell_encode_csr(csr, fmt="fp16", C=C, sigma=1, k_left=0)
        assert e.value.code == 1
        A = ps.packsell_encode_csr(csr, fmt="fp16", C=C, sigma=1)
        assert (A.n_words, A.n_dummies, A.n_pad) == (want.n_words, want.n_dummies, want.n_pad)
        assert (ps.packsell_arrays(A)["pack"] == ps.packsell_arrays(want)["pack"]).all()
