"""The level-0 encoder's parse graph at the limit of its tables, on the host."""
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
    tmp = tmp_path_factory.mktemp("nodecap")
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    obj, out = tmp / "oracle.o", tmp / "node_cap_test"
    subprocess.check_call(["gcc", "-O2", "-ffp-contract=off", "-std=c99", "-c",
                           os.path.join(ROOT, "oracle", "oracle.c"), "-o", str(obj)])
    subprocess.check_call(["g++", "-std=c++20", "-O1", "-pthread", "-x", "c++", "-I", cuda_inc,
                           os.path.join(HERE, "host_emu", "node_cap_test.cu"), "-x", "none",
                           str(obj), "-o", str(out), "-lm"])
    return str(out)


# the kernels of a fixed block size have larger tables
@pytest.mark.parametrize("size,nodes", [(1024, 0), (2048, 96), (8192, 320), (4096, 0), (8192, 0),
                                        (16384, 0)])
def test_blocks_around_the_node_limit(exe, size, nodes):
    r = subprocess.run([exe, str(size), str(nodes)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
