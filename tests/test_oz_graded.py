"""Host check that the FP64 contraction on the FP16 tensor cores is as accurate as
an FMA chain for rows and columns of any scaling (csrc/oz_digits.h: which results
of the digit products are taken, tests/oz_graded_check.cpp)."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1905_01180_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "oz_graded_check.cpp")


def test_graded_dot_products(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "oz_graded_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, SRC, "-o", exe],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=600).stdout
    vals = {k: int(v) for k, v in re.findall(r"^(\w+) (-?\d+)", out, flags=re.M)}
    # rms error over sum |x y|, relative to the FMA chain's (which is 0.45 2^-53 and more), per length and
    # spread of the exponents: the criterion bounds the worst accepted one by 3.3 2^-53, a factor of 7
    rms = {k: v for k, v in vals.items() if k.startswith("rms_")}
    assert len(rms) == 64 and max(rms.values()) <= 7_000_000, out
    assert all(v <= 2_000_000 for k, v in rms.items() if int(k.split("_")[1]) >= 20), out
    # on well scaled vectors of the usual lengths the digits do the work, at less than the chain's error
    for K in (20, 33, 48, 66, 96):
        assert vals[f"taken_{K}_0"] >= 999_000 and vals[f"rms_{K}_0"] <= 1_000_000, out
    assert vals["over_bound"] == 0 and vals["wrong"] == 0, out
