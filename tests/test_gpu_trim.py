"""packsell_trim returns the memory that the library keeps after its matrices are gone."""
import gc

import pytest

from paper_2604_13433_gb300 import inputs as I

from _gpu import P, need_gpu, torch

pytestmark = pytest.mark.gpu


def test_trim_returns_what_destroyed_matrices_held():
    need_gpu()
    ps = P()
    csr = I.stencil27(96, seed=1)
    ps.packsell_trim()
    A = ps.packsell_encode_csr(csr, fmt="fp16", D=15)
    held = 4 * A.n_words  # about 94 MB
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    with_matrix = torch.cuda.mem_get_info()[0]
    del A
    gc.collect()
    ps.packsell_trim()
    assert torch.cuda.mem_get_info()[0] >= with_matrix + held // 2
