"""Host checks of the sliced graphs the decode kernels walk and of their
shared-memory layout, built with g++ (tests/slice_check.cpp states the
invariants): the codes, window shapes and options decoded elsewhere, small and
degenerate codes, and sizes around a slice's 32 nodes."""
import os
import shutil
import subprocess

import pytest

from paper_2403_18901_gb300.workloads import CODES

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "..", "paper_2403_18901_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cxx, inc = shutil.which("g++"), "/usr/local/cuda/include"
    if cxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path_factory.mktemp("slices") / "slice_check")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + inc, "-o", exe, os.path.join(HERE, "slice_check.cpp"),
                    os.path.join(SRC, "dem_host.cpp")], check=True, capture_output=True)
    return exe


def _code(key):
    c = CODES[key]
    return [c["l"], c["m"]] + [v for t in c["A"] + c["B"] for v in t]


ONE = [1, 1] + [0] * 12
SMALL = [4, 4, 1, 0, 0, 1, 2, 2, 0, 1, 1, 0, 3, 2]      # w = 16: half a slice of checks per block
ODD = [11, 3, 3, 0, 0, 1, 7, 2, 0, 1, 1, 0, 5, 2]       # w = 33: one check past a slice
# (code, rounds (0: code capacity), W, F, merge_h1, shorten)
CASES = [(_code("72"), 6, 3, 1, 0, 1), (_code("90"), 10, 2, 1, 0, 1), (_code("108"), 10, 4, 1, 0, 1),
         (_code("144"), 12, 3, 1, 0, 1), (_code("144"), 12, 5, 2, 0, 1), (_code("144"), 5, 3, 1, 1, 1),
         (_code("144"), 5, 3, 1, 2, 1), (_code("288"), 4, 4, 1, 0, 1), (_code("72"), 4, 3, 1, 0, 0),
         (_code("288"), 0, 1, 1, 0, 0), (ONE, 2, 1, 1, 0, 1), (ONE, 3, 2, 1, 0, 0), (SMALL, 3, 2, 1, 0, 1),
         (ODD, 3, 1, 1, 0, 1), (ODD, 4, 3, 1, 0, 1)]


@pytest.mark.parametrize("code,rounds,W,F,merge,shorten", CASES)
def test_slices_and_layout(checker, code, rounds, W, F, merge, shorten):
    args = [str(v) for v in code + [rounds, W, F, merge, shorten, 40]]
    r = subprocess.run([checker] + args, capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", (args, r.stdout, r.stderr)
