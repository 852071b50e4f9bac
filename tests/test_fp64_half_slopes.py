"""The FP64 half slopes of the kernels and the slope multipliers of the adjoint
follow the limiter's definition (a host build of the kernels' own headers)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_half_slopes_and_adjoint_multipliers(tmp_path):
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = cand if os.path.exists(cand) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "half_slopes_check")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", os.path.join(HERE, "half_slopes_check.cu"),
                           "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
