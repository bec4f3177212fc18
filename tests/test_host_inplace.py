"""The in-place LZ4 decoders of csrc/ compiled for the host, on corrupt
blocks whose output would run into the input still to be read."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("CUDA toolkit not available")
    tmp = tmp_path_factory.mktemp("inplace")
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    obj, out = tmp / "oracle.o", tmp / "inplace_bound_test"
    subprocess.check_call(["gcc", "-O2", "-ffp-contract=off", "-std=c99", "-c",
                           os.path.join(ROOT, "oracle", "oracle.c"), "-o", str(obj)])
    subprocess.check_call(["g++", "-std=c++20", "-O1", "-pthread", "-x", "c++", "-I", cuda_inc,
                           os.path.join(HERE, "host_emu", "inplace_bound_test.cu"), "-x", "none",
                           str(obj), "-o", str(out), "-lm"])
    return str(out)


@pytest.mark.parametrize("size,phase", [(8192, 3), (16384, 0), (65536, 15)])
def test_output_never_passes_the_unread_input(exe, size, phase):
    r = subprocess.run([exe, str(size), str(phase)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
