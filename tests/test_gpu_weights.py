"""GPU tests of the learned weights' ordering for the pre-BP (bit-exact decoding
with weights itself is in test_gpu_parity): weights changed in place or replaced
by others of another length, weights installed in some windows only, and batches
whose members have weights, have them in some windows, or have none, installed
before and after the batch was made.  Every result equals that of a fresh
decoder with the same weights, decoded window by window."""
import pytest

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


def _weights(dec, windows, T, seed):
    gen = torch.Generator().manual_seed(seed)
    return {k: (0.45 + 0.45 * torch.rand((T, dec.window_info(k)["n_edges"]), generator=gen)).cuda() for k in windows}


def _decoder(key, R, W, n, weights=None):
    dem = qdec.Dem(CODES[key], 0.004, R)
    dec = qdec.Decoder(dem, preset("configured", k_guess=3, p=0.004, W=W), max_shots=n)
    for k, w in (weights or {}).items():
        dec.set_weights(k, w)
    return dem, dec


def _decode(dec, det0, n, mode=1):
    dec.set_launch(mode)
    det = det0.clone()
    corr = torch.zeros((n, dec.corr_words), dtype=torch.int32, device="cuda")
    pred = torch.zeros(n, dtype=torch.int32, device="cuda")
    resid = torch.zeros(n, dtype=torch.int32, device="cuda")
    for k in range(dec.n_windows):
        dec.decode_window(k, det, n, corr)
        dec.commit(k, corr, n, det, pred, resid)
    torch.cuda.synchronize()
    return [x.cpu() for x in (det, pred, resid)]


def _same(a, b):
    return all(torch.equal(x, y.cpu()) for x, y in zip(a, b))


@pytest.mark.parametrize("key,R,W,T,T2,mode", [("72", 6, 3, 1, 25, 1), ("72", 6, 3, 25, 3, 2), ("144", 4, 3, 7, 12, 1),
                                              ("90", 4, 2, 12, 30, 3)])
def test_replaced_weights(key, R, W, T, T2, mode):
    n = 20
    dem, dec = _decoder(key, R, W, n)
    det0, _ = dem.sample(31, 0, n)
    plain = _decode(dec, det0, n, mode)
    w = _weights(dec, range(dec.n_windows), T, 1)
    for k in w:
        dec.set_weights(k, w[k])
    first = _decode(dec, det0, n, mode)
    assert _same(first, _decode(_decoder(key, R, W, n, w)[1], det0, n, mode))
    for k in w:  # in place
        w[k].mul_(1.125)
    assert _same(_decode(dec, det0, n, mode), _decode(_decoder(key, R, W, n, w)[1], det0, n, mode))
    w2 = {**w, **_weights(dec, range(1, dec.n_windows, 2), T2, 2)}  # another length in every second window
    for k in w2:
        dec.set_weights(k, w2[k])
    assert _same(_decode(dec, det0, n, mode), _decode(_decoder(key, R, W, n, w2)[1], det0, n, mode))
    for k in w2:
        dec.set_weights(k, None)
    assert _same(_decode(dec, det0, n, mode), plain)


@pytest.mark.parametrize("after", [False, True])
def test_batch_of_members_with_and_without_weights(after):
    shapes = [("72", 6, 2, 40), ("90", 6, 3, 30), ("72", 6, 3, 30), ("108", 6, 3, 20)]
    mem, want = [], []
    for i, (key, R, W, n) in enumerate(shapes):
        dem, dec = _decoder(key, R, W, n)
        windows = [range(dec.n_windows), [1], [], [0]][i]  # all, some, none, the first
        w = _weights(dec, windows, 9, 50 + i)
        det, _ = dem.sample(700 + i, 0, n)
        want.append(_decode(_decoder(key, R, W, n, w)[1], det, n))
        mem.append((dec, det, n, w))
    batch = qdec.Batch([m[0] for m in mem]) if after else None
    for dec, _, _, w in mem:
        for k in w:
            dec.set_weights(k, w[k])
    batch = batch or qdec.Batch([m[0] for m in mem])
    det = [m[1].clone() for m in mem]
    n = [m[2] for m in mem]
    pred = [torch.zeros(x, dtype=torch.int32, device="cuda") for x in n]
    resid = [torch.zeros(x, dtype=torch.int32, device="cuda") for x in n]
    for j in range(batch.n_steps):
        batch.step(j, det, n, pred, resid)
    torch.cuda.synchronize()
    for i, got in enumerate(zip(det, pred, resid)):
        assert _same(want[i], got), i
