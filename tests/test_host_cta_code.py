"""The CTA-wide transpose and level-0 LZ4 encoder of csrc/ compiled for the
host (one thread per CUDA thread) against the oracle and the one-warp encoder."""
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
    tmp = tmp_path_factory.mktemp("cta")
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    obj, out = tmp / "oracle.o", tmp / "cta_code_test"
    subprocess.check_call(["gcc", "-O2", "-ffp-contract=off", "-std=c99", "-c",
                           os.path.join(ROOT, "oracle", "oracle.c"), "-o", str(obj)])
    subprocess.check_call(["g++", "-std=c++20", "-O1", "-pthread", "-x", "c++", "-I", cuda_inc,
                           os.path.join(HERE, "host_emu", "cta_code_test.cu"), "-x", "none",
                           str(obj), "-o", str(out), "-lm"])
    return str(out)


# blocks of one word to 64 KiB: full ones, and shortened ones whose bit-rows
# are no whole words; kinds 0 walk, 1-2 stretches, 3 more matches than the
# tables hold nodes
SHAPES = [(4, 2048), (4, 1024), (4, 1008), (4, 8), (4, 1304), (4, 16384), (4, 3072), (8, 1024), (8, 512),
          (8, 200), (8, 4096), (2, 4096), (2, 2048), (2, 2008), (2, 96), (1, 8192), (1, 4096),
          (1, 4104), (1, 128), (1, 24)]


@pytest.mark.slow
@pytest.mark.parametrize("es,n,kind", [(es, n, k) for es, n in SHAPES for k in range(4)
                                       if es * n <= 8192 or k == 1])
def test_cta_code_on_host(exe, es, n, kind):
    r = subprocess.run([exe, str(es), str(n), str(kind), str(7 * n + kind)], capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
