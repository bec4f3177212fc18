"""The float32 shortcut to the full covariance's q, compiled for the host,
against the quotient in 64 bits over every accepted magnitude."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_float32_q_has_the_granularity_of_the_64_bit_q(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("CUDA toolkit not available")
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    exe = tmp_path / "full_q_test"
    subprocess.check_call(["g++", "-std=c++20", "-O1", "-ffp-contract=off", "-x", "c++", "-I", cuda_inc,
                           os.path.join(HERE, "host_emu", "full_q_test.cu"), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
