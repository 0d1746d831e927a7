"""The training GEMM's output pieces (csrc/tc_common.cuh), compiled for the host: its
tiles are a multiple of 16 columns wide, and an output whose width is not (8, 24,
72, 80 columns ...) has pieces beyond its last column, which must not be stored."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_gemm_pieces_stay_inside_the_output(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "gemm_pieces_check"
    src = os.path.join(ROOT, "tests", "host", "gemm_pieces_check.cu")
    inc = [os.path.join(ROOT, "paper_2601_08266_gb300", "csrc"), os.path.join(ROOT, "include")]
    subprocess.run([nvcc, "-std=c++17", "-O2", "-arch=sm_103a", "-x", "cu", *[f"-I{p}" for p in inc],
                    src, "-o", str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout + r.stderr
