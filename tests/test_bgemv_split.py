"""How the block product deals out its row blocks (csrc/gemv_split.h): the host check compiles
the rule and holds it against sizes at which one form was measured to be faster."""
import pathlib
import shutil
import subprocess

import pytest

ROOT = pathlib.Path(__file__).resolve().parents[1]


def test_rule(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = tmp_path / "bgemv_split_check"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", str(ROOT / "paper_1511_07207_gb300" / "csrc"),
                    str(ROOT / "tests" / "bgemv_split_check.cpp"), "-o", str(exe)], check=True)
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stdout
    assert "mismatches 0" in p.stdout
