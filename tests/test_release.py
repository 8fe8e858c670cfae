"""A destroyed matrix's memory goes back only after its own device has finished
(``csrc/release.h``), checked on a stand-in for the CUDA runtime: with another
device current, with a device that cannot be waited for, and with one that
cannot be selected."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2604_13433_gb300", "csrc")


def test_memory_goes_back_after_its_device_has_finished(tmp_path):
    exe = str(tmp_path / "release_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-Wno-format-security", "-pthread",
                    "-I", CSRC, os.path.join(HERE, "release_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
