"""Run in a child process by test_gpu_checks_backward.py, with PACKSELL_CHECKS=1.

A padding word of a slice of 32 rows is rewritten as a word with the flag, no
delta and the value 0: its column stays the row's last one, but the row now
carries one value more than its row pointer has room for. The products that
write the pattern's values skip that write and packsell_check_status reports
the position; every other value is the valid matrix's. The row is not the last
one, so even an unchecked write would stay inside the output. Prints
"checks ok" on success."""
import os
import sys

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from paper_2604_13433_gb300 import build, inputs as I  # noqa: E402

assert os.environ.get("PACKSELL_CHECKS") == "1"
build.build(checks=True)
from paper_2604_13433_gb300 import packsell as ps  # noqa: E402

assert ps.lib().packsell_checks_build() == 1

csr = I.random_csr(500, 400, 0.03, seed=7, empty_rows=0.05)
A = ps.packsell_encode_csr(csr, fmt="fp16", D=15, C=32, sigma=1, keep_rowptr=True)
x = torch.from_numpy(I.uniform(csr.m, seed=3)).cuda()
dy = torch.from_numpy(I.uniform(csr.n, seed=4)).cuda()


def status():
    code = ps.lib().packsell_check_status(A.handle, None)
    return code, ps.lib().packsell_last_error().decode()


def products():
    _, dval = ps.packsell_spmv_backward(A, x, dy, need_dx=True, need_dval=True)
    first = status()
    outer = ps.packsell_pattern_outer(A, 1.0, dy, x)
    return dval.cpu().numpy(), first, outer.cpu().numpy(), status()


good, s1, good_outer, s2 = products()
assert s1 == (0, "") and s2 == (0, ""), (s1, s2)
row_of = np.repeat(np.arange(csr.n), np.diff(csr.rowptr))
want = dy.cpu().numpy()[row_of] * x.cpu().numpy()[csr.col]
assert np.array_equal(good, want) and np.array_equal(good_outer, want)

arr = ps.packsell_arrays(A)
pack, offset = arr["pack"], arr["offset"]
for row in range(100, csr.n - 40):  # a filled row that ends in padding
    k, l = divmod(row, 32)
    slots = [int(offset[k]) + j * 32 + l for j in range(int(offset[k + 1] - offset[k]) // 32)]
    if csr.rowptr[row + 1] > csr.rowptr[row] and slots and pack[slots[-1]] == 0:
        break
at = min(p for p in slots if pack[p] == 0)


class _View:
    __cuda_array_interface__ = {"shape": (A.n_words,), "typestr": "<i4",
                                "data": (A.info.pack, False), "version": 3}


words = torch.as_tensor(_View(), device="cuda")
words[at] = 1
torch.cuda.synchronize()
dval, s1, outer, s2 = products()
for code, msg in (s1, s2):
    assert code == 11 and f" 1 out-of-range accesses skipped (first index {csr.rowptr[row + 1]})" in msg, (code, msg)
assert np.array_equal(dval, want) and np.array_equal(outer, want)
words[at] = 0
torch.cuda.synchronize()
assert products()[1] == (0, "")
print("checks ok")
