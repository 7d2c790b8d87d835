"""The packed hard-sphere trials (library code in
paper_1503_00707_gb300/csrc/hs.cpp, compiled into a small checker with g++):
read back the way the gather kernel reads them, every node's weighted trials
come back whole, at the smallest and largest grids, at trial counts that give a
node from one to all lanes of a warp, and with partly filled warps and CTAs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe, lib = str(tmp_path_factory.mktemp("pack") / "check"), os.path.join(CUDA, "lib64")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-pthread", "-I", os.path.join(CUDA, "include"),
                           os.path.join(ROOT, "tests", "hs_pack_check.cpp"), "-o", exe, "-L", lib, "-lcudart",
                           "-Wl,-rpath," + lib])
    return exe


@pytest.mark.parametrize("nv, M", [(32, 32), (32, 1024), (130, 256), (512, 64), (1728, 512), (4096, 128), (14336, 32)])
def test_packed_trials(checker, nv, M):
    out = subprocess.run([checker, str(nv), str(M)], capture_output=True, text=True, timeout=600, check=True).stdout.split()
    assert int(out[0]) == 0
    if (nv, M) == (4096, 128):
        # values gathered per wavefront of 32: 24 and 23 on these tables, 20 without the local search
        assert float(out[1]) > 22 and float(out[2]) > 21.5
