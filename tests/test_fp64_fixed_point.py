"""The fixed-point FP64 reciprocal and square root are within 0.51 ulp (a host
build of the kernels' own header against long double; the bound is half an
ulp of rounding plus the documented 2^-61 truncation)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fixed_point_reciprocal_and_root(tmp_path):
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = cand if os.path.exists(cand) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "fixed_point_check")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", os.path.join(HERE, "fixed_point_check.cu"),
                           "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
