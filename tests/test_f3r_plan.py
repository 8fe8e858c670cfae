"""Which form an Arnoldi step of F3R takes (``csrc/f3r_plan.h``): the sizes where
the rule changes on 152 SMs at four blocks each, an unknown occupancy, and a
device that grants fewer blocks than it reports, where the separate kernels run."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2604_13433_gb300", "csrc")
ALL = 608  # 152 SMs, four blocks each; 256 threads hold 4 to 32 elements
CASES = [  # n, SMs, blocks per SM (16, 32 elements), blocks granted -> elements, blocks, trial launches
    ((1, 152, 4, 4, ALL), (16, 1, 1)),
    ((1024, 152, 4, 4, ALL), (16, 1, 1)),
    ((1028, 152, 4, 4, ALL), (16, 2, 1)),
    ((4 * ALL * 256, 152, 4, 4, ALL), (16, ALL, 1)),
    ((16 * ALL * 256 + 3, 152, 4, 4, ALL), (16, ALL, 1)),
    ((16 * ALL * 256 + 4, 152, 4, 4, ALL), (32, ALL, 1)),
    ((32 * ALL * 256 + 3, 152, 4, 4, ALL), (32, ALL, 1)),
    ((32 * ALL * 256 + 4, 152, 4, 4, ALL), (0, 0, 0)),
    ((1000000, 152, 5, 5, ALL), (16, ALL, 1)),
    ((1000000, 152, 0, 4, ALL), (32, ALL, 1)),
    ((1000000, 152, 0, 0, ALL), (0, 0, 0)),
    ((1000000, 152, 4, 4, ALL - 1), (0, 0, 2)),  # fewer SMs granted than reported
    ((100000, 152, 4, 4, ALL - 1), (16, 98, 1)),
    ((100000, 152, 4, 4, 0), (0, 0, 2)),         # no cooperative launch at all
]


def test_form_of_an_arnoldi_step(tmp_path):
    exe = str(tmp_path / "f3r_plan_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC,
                    os.path.join(HERE, "f3r_plan_check.cpp"), "-o", exe], check=True)
    args = [str(v) for case, _ in CASES for v in case]
    out = subprocess.run([exe, *args], capture_output=True, text=True, check=True).stdout
    got = [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    assert got == [want for _, want in CASES]
