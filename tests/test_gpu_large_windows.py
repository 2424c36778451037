"""GPU parity of windows whose shortened graph does not fit shared memory next to
what always lies there, so that its entries go to the CTA's region of global
memory with the path states: unshortened windows of 17 rounds, and of 13 with
learned weights (whose edge ids count too).  Bit-exact against the oracle."""
import numpy as np
import pytest

from conftest import oracle_dem
from test_gpu_parity import _pipeline
from paper_2403_18901_gb300 import build as qbuild
from paper_2403_18901_gb300 import qdec
from paper_2403_18901_gb300.workloads import CODES, preset

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qbuild.build()
    qdec.lib()


@pytest.mark.parametrize("key,W,k,mode", [("72", 17, 4, 0), ("72", 17, 3, 3), ("144", 9, 2, 1)])
def test_unshortened(key, W, k, mode):
    params = preset("configured", k_guess=k, W=W, shorten=0, n_pre=20, d_max_main=12)
    _pipeline(key, W, 0.003, params, n=6, seed=170 + W, trace_windows=(0,), mode=mode)


def test_learned_weights():
    W, n = 13, 6
    params = preset("configured", k_guess=3, W=W, shorten=0, n_pre=20, d_max_main=12)
    ne = oracle_dem("72", 0.003, W).window(W, 1, 1)["n_edges"]
    rng = np.random.default_rng(8)
    weights = {1: rng.uniform(0.45, 0.9, size=(15, ne)).astype(np.float32)}
    _pipeline("72", W, 0.003, params, n=n, seed=188, trace_windows=(1,), mode=0, weights=weights)


@pytest.mark.parametrize("ranker,mode", [(False, 0), (True, 2)])
def test_path_mode_with_edge_ids_in_global_memory(ranker, mode):
    """One size at which learned weights' edge ids are what does not fit a path's CTA."""
    W, n = 10, 4
    params = preset("configured", k_guess=3, W=W, shorten=0, n_pre=20, d_max_main=12)
    o = oracle_dem("72", 0.003, W)
    rng = np.random.default_rng(8)
    weights = {k: rng.uniform(0.45, 0.9, size=(15, o.window(W, 1, k)["n_edges"])).astype(np.float32) for k in range(2)}
    rk = None
    if ranker:
        rk = np.zeros(641, np.float32)
        rk[:512] = rng.normal(0, 0.6, 512)
        rk[576:640] = rng.normal(0, 0.5, 64)
    dec = qdec.Decoder(qdec.Dem(CODES["72"], 0.003, W), params, max_shots=n)
    for k, w in weights.items():
        dec.set_weights(k, torch.from_numpy(w).cuda())
    assert dec.launch_info(0)["path_smem"] <= 232448 < dec.launch_info(0)["shot_smem"]
    _pipeline("72", W, 0.003, params, n=n, seed=191, trace_windows=(0, 1), mode=mode, weights=weights, ranker=rk)


def test_removing_the_weights_brings_the_smaller_layout_back():
    W, n = 13, 4
    dem = qdec.Dem(CODES["72"], 0.003, W)
    dec = qdec.Decoder(dem, preset("configured", k_guess=3, W=W, shorten=0, n_pre=20, d_max_main=8), max_shots=n)
    before = dec.launch_info(0)
    det, _ = dem.sample(5, 0, n)
    corr = [torch.zeros((n, dec.corr_words), dtype=torch.int32, device="cuda") for _ in range(2)]
    dec.decode_window(0, det, n, corr[0])
    dec.set_weights(0, torch.full((3, dec.window_info(0)["n_edges"]), 0.625, device="cuda"))
    dec.decode_window(0, det, n, corr[1])  # every weight is the normalisation
    assert torch.equal(*corr)
    dec.set_weights(0, None)
    assert dec.launch_info(0) == before
    corr[1].zero_()
    dec.decode_window(0, det, n, corr[1])
    assert torch.equal(*corr)
