"""The fixed-point hop of the FP64 and double-float dslash, compiled for the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_hop_host_side(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "fix")
    csrc = os.path.join(ROOT, "paper_1106_4964_gb300", "csrc")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-I", csrc, os.path.join(ROOT, "tests", "dslash_fix_check.cu"),
                           "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
