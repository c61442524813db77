"""The element means' division by three without a division (csrc/element_mean.h, compiled here with the host
compiler; the same products and fused multiply-adds as on the GPU, each rounded once) is the division, bit for
bit."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("seed", [1, 2])
def test_third_of_a_sum_is_the_division(tmp_path, seed):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "element_mean_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-Wall", "-Werror",
                    "-I", os.path.join(ROOT, "paper_2403_04491_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "c", "element_mean_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe, "1000000", str(seed)], capture_output=True, text=True, check=True).stdout
    assert out.split()[-1] == "0", out
