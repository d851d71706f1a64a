"""The LU panel kernel whose rows lie in global memory (tests/lu_panel_check.cu, compiled here
with the library's flags)."""
import pathlib
import subprocess

import pytest

from paper_1511_07207_gb300 import build

pytestmark = pytest.mark.gpu

ROOT = pathlib.Path(__file__).resolve().parents[1]


def test_rows_in_global_memory(gpu, tmp_path):
    exe = tmp_path / "lu_panel_check"
    subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS + [str(ROOT / "tests" / "lu_panel_check.cu"), "-o", str(exe)],
                   check=True, timeout=300)
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stdout
    assert "mismatches 0" in p.stdout
