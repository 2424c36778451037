"""GPU parity of the ranking's selection (Sec. III: the first 2w' columns by
the four-iteration sum, ties by column): keys that are all prior sums and so
mostly equal (no pre-BP), few distinct keys (one iteration), and windows whose
column counts lie on either side of a power of two, in every launch shape.
Exact comparison of the short columns and everything after them, as in
test_gpu_parity."""
import pytest

from paper_2403_18901_gb300 import build as qbuild
from paper_2403_18901_gb300 import qdec
from paper_2403_18901_gb300.workloads import preset
from test_gpu_parity import _pipeline

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qbuild.build()
    qdec.lib()


@pytest.mark.parametrize("key,R,W,n_pre,mode", [("72", 4, 1, 0, 1), ("72", 4, 2, 1, 1), ("144", 4, 3, 0, 1),
                                               ("90", 4, 2, 3, 2), ("144", 4, 2, 0, 2), ("108", 4, 3, 1, 3),
                                               ("288", 3, 2, 2, 1)])
def test_selection_with_equal_keys(key, R, W, n_pre, mode):
    params = preset("configured", k_guess=2, W=W, n_pre=n_pre, d_max_main=6)
    _pipeline(key, R, 0.003, params, n=24, seed=9000 + R + W, trace_windows=(0, 1), mode=mode)
