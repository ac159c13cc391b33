"""Sums of FP32 values in three FP32 values (csrc/fp32_sum.cuh) on the host: rounded once (a unit in the last place of
FP64 is 2^-52, half of it the bound), never further from the exact sum than FP64 additions, and marked by a value that is not
finite where FP32's range ends (tests/fp32_sum_host.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_less_exact_than_fp64(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    exe = str(tmp_path / "fp32_sum")
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", os.path.join(ROOT, "paper_1708_01663_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fp32_sum_host.cpp"), "-o", exe], check=True)
    worst, further, finite = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    assert float(worst) <= 1.0 and further == "0" and finite == "0"
