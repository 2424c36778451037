"""GPU test of batched steps with members whose window does not fit the step's
shape in slices although its plain arrays do (unshortened windows with learned
weights at one size per code), so that they are decoded by a launch of their own:
a batch of such members only, one beside small windows, and weights installed
after the batch was made.  Equal to decoding every member by itself."""
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


def _member(W, n, weights, seed, shorten=0):
    dem = qdec.Dem(CODES["72"], 0.004, W)
    params = preset("configured", k_guess=4, p=0.004, W=W, shorten=shorten, n_pre=20, d_max_main=12)
    dec = qdec.Decoder(dem, params, max_shots=n)
    gen = torch.Generator().manual_seed(seed)
    w = {k: (0.45 + 0.45 * torch.rand((9, dec.window_info(k)["n_edges"]), generator=gen)).cuda()
         for k in range(dec.n_windows)} if weights else {}
    det, _ = dem.sample(seed, 0, n)
    return dict(dec=dec, n=n, w=w, det=det)


def _install(m):
    for k, w in m["w"].items():
        m["dec"].set_weights(k, w)


def _alone(m):
    n, dec = m["n"], m["dec"]
    det = m["det"].clone()
    corr = torch.zeros((n, dec.corr_words), dtype=torch.int32, device="cuda")
    pred, resid = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    for k in range(dec.n_windows):
        dec.decode_window(k, det, n, corr)
        dec.commit(k, corr, n, det, pred, resid)
    torch.cuda.synchronize()
    return [x.cpu() for x in (det, pred, resid)]


# members (W, shots, weights, shorten); CTAs per SM of every step (0: the default shape)
@pytest.mark.parametrize("shape,ctas,after", [([(5, 30, True, 0)], 2, False),
                                              ([(3, 200, False, 1), (5, 30, True, 0)], 2, False),
                                              ([(3, 200, False, 1), (5, 30, True, 0)], 0, True),
                                              ([(3, 200, False, 1), (10, 12, True, 0)], 0, False)])
def test_members_that_do_not_fit_the_shape(shape, ctas, after):
    mem = [_member(W, n, w, 90 + i, s) for i, (W, n, w, s) in enumerate(shape)]
    batch = qdec.Batch([m["dec"] for m in mem]) if after else None
    for m in mem:
        _install(m)
    want = [_alone(m) for m in mem]
    batch = batch or qdec.Batch([m["dec"] for m in mem])
    det = [m["det"].clone() for m in mem]
    n = [m["n"] for m in mem]
    pred, resid = ([torch.zeros(x, dtype=torch.int32, device="cuda") for x in n] for _ in range(2))
    for j in range(batch.n_steps):
        if ctas:
            batch.set_shape(j, 8, ctas)
        batch.step(j, det, n, pred, resid)
    torch.cuda.synchronize()
    for x, *got in zip(want, det, pred, resid):
        assert all(torch.equal(a, b.cpu()) for a, b in zip(x, got))
