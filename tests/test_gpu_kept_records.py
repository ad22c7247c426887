"""Records of the on-chip cycles' lowest diagonals (tests/kept_records_check.cu)."""
import os
import subprocess

import pytest

from paper_1907_12334_gb300 import build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1907_12334_gb300", "csrc")


def test_diagonals_are_the_sums_of_the_faces(tmp_path):
    exe = tmp_path / "kept_records_check"
    cmd = [build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.INCLUDE, "-I", CSRC,
           os.path.join(HERE, "kept_records_check.cu"), os.path.join(CSRC, "api.cu"), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:]
