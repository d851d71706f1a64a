"""The direct methods form the products of their rank updates with integer
operations (csrc/mul53.h).  This host check compiles that code and compares
it bit for bit with the rounded FP64 product: random operands over the whole
accepted exponent range and at its borders, exact products, ties (reported,
never guessed), and the borders of the significand's one-bit shift.  The
device form is checked through the factors in test_gpu_lu.py,
test_gpu_cholesky.py and test_gpu_trail.py."""
import pathlib
import shutil
import subprocess

import pytest

ROOT = pathlib.Path(__file__).resolve().parents[1]


def test_mul53_bits_match_the_rounded_product(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = tmp_path / "mul53_check"
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off",
                    "-I", str(ROOT / "paper_1511_07207_gb300" / "csrc"),
                    str(ROOT / "tests" / "mul53_check.cpp"), "-o", str(exe)], check=True)
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert p.returncode == 0, p.stdout
    assert "mismatches 0" in p.stdout
