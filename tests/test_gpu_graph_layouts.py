"""GPU test of CUDA graphs captured before a decoder lays its windows out again
(learned weights or a ranker installed or removed, another launch mode): a replay
gives what it gave at first -- it keeps the layouts, the path schedule and the
buffers of its capture -- and writes into no memory that the decoder has handed
back."""
import numpy as np
import pytest

from paper_2403_18901_gb300 import build as qbuild
from paper_2403_18901_gb300 import qdec
from paper_2403_18901_gb300.workloads import CODES, preset

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,k_guess", [(1, 5), (3, 4), (0, 4)])
def test_replay_after_new_layouts(mode, k_guess):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qbuild.build()
    n, dem = 400, qdec.Dem(CODES["72"], 0.004, 6)
    dec = qdec.Decoder(dem, preset("configured", k_guess=k_guess, p=0.004), max_shots=n)
    dec.set_launch(mode)
    det0, _ = dem.sample(78, 0, n)
    det = det0.clone()
    pred, resid = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    corr = torch.zeros((n, dec.corr_words), dtype=torch.int32, device="cuda")

    def decode(stream=None):
        for k in range(dec.n_windows):
            dec.decode_window(k, det, n, corr, stream=stream)
            dec.commit(k, corr, n, det, pred, resid, stream=stream)

    def outcome(run):
        det.copy_(det0)
        pred.zero_()
        resid.zero_()
        run()
        torch.cuda.synchronize()
        return [x.cpu() for x in (det, pred, resid)]

    rng = np.random.default_rng(2)
    ranker = np.concatenate([rng.normal(0, 0.6, 512), np.zeros(64), rng.normal(0, 0.5, 64), [0]]).astype(np.float32)
    weights = [torch.full((3, dec.window_info(k)["n_edges"]), 0.55, device="cuda") for k in range(dec.n_windows)]

    def set_weights(on):
        for k, w in enumerate(weights):
            dec.set_weights(k, w if on else None)

    steps = [lambda: dec.set_ranker(ranker), lambda: set_weights(True), lambda: dec.set_launch(3),
             lambda: dec.set_ranker(None), lambda: dec.set_launch(mode), lambda: set_weights(False)]
    first = outcome(decode)
    s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        decode(s)
    for i, step in enumerate(steps):
        step()
        torch.cuda.empty_cache()
        taken = [torch.full((1 << 22,), 0x5A5A5A5A, dtype=torch.int32, device="cuda") for _ in range(32)]
        second = outcome(decode)
        assert all(torch.equal(a, b) for a, b in zip(first, outcome(graph.replay))), i
        assert all(int((x != 0x5A5A5A5A).sum()) == 0 for x in taken), i
        assert all(torch.equal(a, b) for a, b in zip(second, outcome(decode))), i
        del taken
    assert all(torch.equal(a, b) for a, b in zip(first, second))
