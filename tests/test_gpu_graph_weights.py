"""GPU test of CUDA graphs captured before a decoder's learned weights are replaced:
by others of the same length, by longer ones (whose copy in the pre-BP's order
needs a larger buffer) and by none.  A replay gives what it gave at first, and
writes into no memory that the decoder has handed back."""
import pytest

from paper_2403_18901_gb300 import build as qbuild
from paper_2403_18901_gb300 import qdec
from paper_2403_18901_gb300.workloads import CODES, preset

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2])
def test_replay_after_weights_are_replaced(mode):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qbuild.build()
    n, dem = 24, qdec.Dem(CODES["72"], 0.004, 6)
    dec = qdec.Decoder(dem, preset("configured", k_guess=3, p=0.004), max_shots=n)
    dec.set_launch(mode)
    det0, _ = dem.sample(77, 0, n)
    det = det0.clone()
    pred, resid = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    corr = torch.zeros((n, dec.corr_words), dtype=torch.int32, device="cuda")
    gen = torch.Generator().manual_seed(5)

    def install(T):
        w = [(0.4 + 0.5 * torch.rand((T, dec.window_info(k)["n_edges"]), generator=gen)).cuda()
             for k in range(dec.n_windows)]
        for k, x in enumerate(w):
            dec.set_weights(k, x)
        return w

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

    kept = install(2)  # (the graph reads them)
    first = outcome(decode)
    s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        decode(s)
    for T in (2, 5, 40, 200):
        install(T)
        # memory that a buffer given back would be part of
        torch.cuda.empty_cache()
        taken = [torch.full((1 << 18,), 0x5A5A5A5A, dtype=torch.int32, device="cuda") for _ in range(64)]
        taken += [torch.full((1 << 12,), 0x5A5A5A5A, dtype=torch.int32, device="cuda") for _ in range(256)]
        second = outcome(decode)
        replay = outcome(graph.replay)
        assert all(torch.equal(a, b) for a, b in zip(first, replay)), T
        assert all(int((x != 0x5A5A5A5A).sum()) == 0 for x in taken), T
        assert all(torch.equal(a, b) for a, b in zip(second, outcome(decode))), T
        del taken
    assert kept
