"""Host check of the layouts of windows whose shortened graph, in slices, does
not fit shared memory (tests/large_check.cpp states the invariants): the sizes
at which plain CSC and CSR arrays still fit, per code with and without
shortening, and a smaller window that needs no such layout."""
import os
import shutil
import subprocess

import pytest

from paper_2403_18901_gb300.workloads import CODES

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "..", "paper_2403_18901_gb300", "csrc")
LIMIT = 232448  # dynamic shared memory of a CTA


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cxx, inc = shutil.which("g++"), "/usr/local/cuda/include"
    if cxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path_factory.mktemp("large") / "large_check")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + inc, "-o", exe, os.path.join(HERE, "large_check.cpp"),
                    os.path.join(SRC, "dem_host.cpp")], check=True, capture_output=True)
    return exe


# (code, W, shorten, whether some layout is of this kind)
@pytest.mark.parametrize("key,W,shorten,some", [("72", 17, 0, True), ("72", 11, 0, True), ("72", 52, 1, True),
                                                ("72", 36, 1, True), ("144", 9, 0, True), ("144", 26, 1, True),
                                                ("144", 17, 1, True), ("288", 5, 0, True), ("288", 13, 1, True),
                                                ("72", 10, 0, False), ("90", 8, 0, False), ("108", 7, 0, False),
                                                ("144", 5, 0, False), ("144", 3, 1, False)])
def test_every_window_that_fits_plain_arrays_has_a_layout(checker, key, W, shorten, some):
    c = CODES[key]
    args = [c["l"], c["m"]] + [v for t in c["A"] + c["B"] for v in t] + [W + 1, W, shorten, LIMIT]
    r = subprocess.run([checker] + [str(v) for v in args], capture_output=True, text=True)
    out = r.stdout.split()
    assert r.returncode == 0 and out[0] == "ok", (args, r.stdout, r.stderr)
    assert (int(out[1]) > 0) == some, r.stdout
