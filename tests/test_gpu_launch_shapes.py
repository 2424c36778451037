"""The launch shapes that a batch's size picks -- path mode with 512, 256 or 128
threads, shot mode with one, two or three CTAs per SM -- give the same results:
batches at the edges of each rule against the first shots of one large batch."""
import pytest

from paper_2403_18901_gb300 import build as qbuild
from paper_2403_18901_gb300 import qdec, ranker
from paper_2403_18901_gb300.workloads import CODES, preset

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qbuild.build()
    qdec.lib()


def _windows(dec, det0, n, mode=0):
    dec.set_launch(mode)
    det = det0[:n].clone()
    corr = torch.zeros((n, dec.corr_words), dtype=torch.int32, device="cuda")
    out = []
    for k in range(dec.n_windows):
        status = torch.zeros(n, dtype=torch.int32, device="cuda")
        corr.zero_()
        dec.decode_window(k, det, n, corr, status)
        out += [corr.cpu(), status.cpu()]
        pred, resid = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
        dec.commit(k, corr, n, det, pred, resid)
        out += [pred.cpu(), resid.cpu()]
    return out + [det.cpu()]


def _static(dec, det0, n):
    det = det0[:n].clone()
    pred, resid = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    for k in range(dec.n_windows):
        dec.decode_commit_static(k, det, n, pred, resid)
    torch.cuda.synchronize()
    return det.cpu()


@pytest.mark.parametrize("key,R,W,pre,k,form", [
    ("72", 6, 3, "configured", 3, ""), ("144", 4, 3, "configured", 4, ""), ("144", 4, 3, "paper", 4, ""),
    ("108", 4, 2, "paper", 3, "ranker"), ("90", 4, 3, "configured", 3, "weights"), ("144", 4, 3, "paper", 3, "reuse"),
    ("288", 4, 3, "configured", 4, ""), ("72", 6, 3, "configured", 5, "")])
def test_batch_sizes(key, R, W, pre, k, form):
    dem = qdec.Dem(CODES[key], 0.003, R)
    over = dict(W=W, F=1, **({"reuse_msgs": 1} if form == "reuse" else {}))
    most = 460
    dec = qdec.Decoder(dem, preset(pre, k, 0.003, **over), max_shots=most)
    if form == "ranker":
        dec.set_ranker(ranker.init_params(5).cpu().numpy())
    if form == "weights":
        gen = torch.Generator().manual_seed(3)
        for x in range(dec.n_windows):
            dec.set_weights(x, (0.5 + 0.3 * torch.rand((9, dec.window_info(x)["n_edges"]), generator=gen)).cuda())
    info = dec.launch_info(0)
    sms, nb = info["sms"], 2 ** k + (6 if pre == "paper" else 0)
    det0, _ = dem.sample(91, 0, most)
    want = _windows(dec, det0, most, 1)
    edges = {1, sms // nb, sms // nb + 1, 3 * sms // nb, 3 * sms // nb + 1, 9 * sms // nb,
             9 * sms // nb + 1, 64, 65, sms // 2, sms // 2 + 1, sms, sms + 1, 2 * sms, 2 * sms + 1}
    for n in sorted(e for e in edges if 1 <= e <= most):
        for mode in (0, 2) if n <= 64 else (0,):
            for a, b in zip(_windows(dec, det0, n, mode), want):
                assert torch.equal(a, b[:n]), (n, mode)
        if form != "reuse":  # (whose state carries over between calls)
            assert torch.equal(_static(dec, det0, n), want[-1][:n]), n
