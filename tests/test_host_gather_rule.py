"""The rule that picks the gather of a time-slowest cube, on the host."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_long_time_axes_go_sample_by_sample(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("CUDA toolkit not available")
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    exe = tmp_path / "gather_rule_test"
    subprocess.check_call(["g++", "-std=c++20", "-O1", "-pthread", "-x", "c++", "-I", cuda_inc,
                           os.path.join(HERE, "host_emu", "gather_rule_test.cu"), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
