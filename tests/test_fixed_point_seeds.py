"""The fixed-point FP64 reciprocal and square root are within 0.51 ulp for every
seed error that their derivation allows (relative 2^-21; on the host, with moved
seeds), and on the GPU with the hardware's approximate seeds, which stay inside
that error."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def run(tmp_path, flags, args):
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = cand if os.path.exists(cand) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "fixed_point_seeds_check")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", *flags,
                           os.path.join(HERE, "fixed_point_seeds_check.cu"), "-o", exe])
    r = subprocess.run([exe, *args], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr


def test_moved_seeds(tmp_path):
    run(tmp_path, [], [])


@pytest.mark.gpu
def test_device_seeds(tmp_path):
    run(tmp_path, ["-gencode", "arch=compute_103a,code=sm_103a"], ["gpu"])
