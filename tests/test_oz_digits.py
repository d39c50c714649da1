"""Host check of the digit arithmetic behind the FP64 contraction on the FP16
tensor cores (csrc/oz_digits.h, compiled into the kernels): dot products
through 8-bit digits against double-double sums (tests/oz_digits_check.cpp)."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1905_01180_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "oz_digits_check.cpp")


def test_digit_dot_products(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "oz_digits_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, SRC, "-o", exe],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=600).stdout
    vals = {k: int(v) for k, v in re.findall(r"^(\w+) (-?\d+)", out, flags=re.M)}
    # the a-priori error bound of the splitting holds for every vector
    assert vals["over_bound"] == 0, out
    # every level sum stays below 2^24 (exact in an FP32 accumulator), those of
    # levels 0 - 2 below 2^22, also for the largest digits over the longest window
    assert vals["level_overflow"] == 0, out
    # at least as close to the exact sum as the FP64 FMA chain (rms)
    assert vals["error_ratio_ppm"] <= 1000000, out
    assert vals["one_bad"] == 0, out
    assert vals["special"] == 7, out
