"""Host-side check of the FP32 contraction's choice of tiles (tests/kl_forms_check.cu; no GPU)."""
import os
import shutil
import subprocess

import pytest

from paper_1907_12334_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1907_12334_gb300", "csrc")


def test_no_sm_is_left_without_a_tile(tmp_path):
    nvcc = build.nvcc()
    if not shutil.which(nvcc) and not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "kl_forms_check"
    cmd = [nvcc, *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.INCLUDE, "-I", CSRC,
           os.path.join(HERE, "kl_forms_check.cu"), *(os.path.join(CSRC, f) for f in ("api.cu", "kl_tc.cu")), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:]
