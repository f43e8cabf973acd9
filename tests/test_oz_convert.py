"""The digit arithmetic of the tensor-core FP64 products (csrc/oz_convert.h), bit for bit, on the
host: values into balanced base-256 digits, and 64-bit level sums back into rounded doubles."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_digits_and_sums_match_wide_integers(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "oz_convert_check")
    subprocess.run([cxx, "-O2", "-std=gnu++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1505_02248_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "oz_convert_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe, "300000"], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.startswith("ok ")
