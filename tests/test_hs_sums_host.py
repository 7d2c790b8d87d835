"""The sums of the hard-sphere correction's moment system (library code in
paper_1503_00707_gb300/csrc/hs_sums.cuh, compiled into a small checker with
g++) against extended precision, on cubic, small and the longest grids
(32 nodes an axis, the most that the operator takes).

A thread adds up to 28 terms to a sum, each with a rounding of 2^-48 of it (Sum2)
and a rest of 2^-38 of its values summed with roundings of 2^-24; the threads of a
cell average them out: below 2^-46 (1.4e-14) of the terms' sizes at most, 2^-49
(1.8e-15) in the root mean square.  The sums are also to be no less exact than every
node added by itself in Sum2."""
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
    exe = str(tmp_path_factory.mktemp("sums") / "check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(CUDA, "include"),
                           os.path.join(ROOT, "tests", "hs_sums_check.cpp"), "-o", exe])
    return exe


# nodes of a sign group and threads: 4 x 4 x 8, 8^3, 14 x 16 x 16, 16^3, 24^3, 32 x 10 x 32, 32 x 32 x 24
@pytest.mark.parametrize("half, threads", [((2, 2, 4), 32), ((4, 4, 4), 32), ((7, 8, 8), 128), ((8, 8, 8), 128),
                                           ((12, 12, 12), 128), ((16, 5, 16), 128), ((16, 16, 12), 128)])
def test_sums(checker, half, threads):
    out = subprocess.run([checker, *map(str, half), str(threads)], capture_output=True, text=True, timeout=600,
                         check=True).stdout.splitlines()
    ours, single = ([float(x) for x in line.split()] for line in out)
    assert max(ours[0], ours[2]) < 2.0 ** -46
    assert max(ours[1], ours[3]) < 2.0 ** -49
    assert ours[1] <= single[1] and ours[3] <= single[3]
