"""The kernel names that bench.py reports for SpMM follow the library's dispatch (CPU only)."""
import importlib.util
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _bench():
    spec = importlib.util.spec_from_file_location("bench_kernels_mod", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


@pytest.mark.parametrize("C,k,width,name", [
    (32, 16, 27, "k_spmm_wide"), (32, 64, 48, "k_spmm_wide"), (32, 16, 49, "k_spmm_packed"),
    (32, 64, 4097, "k_spmm_packed"), (32, 4, 27, "k_spmm_packed"), (16, 16, 27, "k_spmm_packed"),
    (1, 16, 4097, "k_split_multi"), (1, 64, 4097, "k_split_rows")])
def test_spmm_kernel_names(C, k, width, name):
    assert _bench().spmm_kernel(C, k, width) == name


def test_width_limit_is_the_dispatchs():
    src = open(os.path.join(ROOT, "paper_2604_13433_gb300", "csrc", "spmm.cu")).read()
    assert re.findall(r"A\.max_width <= (\d+)", src) == ["48"]
