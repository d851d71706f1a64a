"""How the matrix-vector product deals out its tiles (csrc/gemv_split.h): by the work of
the longest CTA against the cost of meeting, not by the number of rows alone.
The host check compiles the rule that the kernel uses; the values and the time of wide
products are checked in test_gpu_gemv_wide.py."""
import pathlib
import shutil
import subprocess

import pytest

ROOT = pathlib.Path(__file__).resolve().parents[1]


def test_rule(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = tmp_path / "gemv_split_check"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", str(ROOT / "paper_1511_07207_gb300" / "csrc"),
                    str(ROOT / "tests" / "gemv_split_check.cpp"), "-o", str(exe)], check=True)
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stdout
    assert "mismatches 0" in p.stdout
