"""GPU test of the training kernel's forward pass with weights that are not finite:
the posteriors of a few iterations equal, bit for bit, the same model in numpy's
FP32 (explicit messages; sums in ascending check order; comparisons that leave a
NaN out).  One edge in two hundred has such a weight, first edges and edges of
every degree among them."""
import numpy as np
import pytest

from paper_2403_18901_gb300 import build as qbuild
from paper_2403_18901_gb300 import qdec
from paper_2403_18901_gb300.workloads import CODES, preset

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _posteriors(win, w, synd, clip):
    f = np.float32
    cp, cr = win["col_ptr"], win["col_rows"]
    col = np.repeat(np.arange(win["n_cols"]), np.diff(cp))
    rows = [np.nonzero(cr == j)[0] for j in range(win["n_rows"])]
    v2c, post = win["llr"][col].astype(f), None
    for wt in w:
        c2v = np.zeros(win["n_edges"], f)
        for j, es in enumerate(rows):
            m1, m2, first, neg = f(np.inf), f(np.inf), -1, int(synd[j])
            for e in es:
                a = abs(v2c[e])
                if a < m1:
                    m1, m2, first = a, m1, e
                elif a < m2:
                    m2 = a
                neg ^= int(v2c[e] < 0)
            for e in es:
                mag = wt[e] * (m2 if e == first else m1)
                c2v[e] = -mag if neg ^ int(v2c[e] < 0) else mag
        post = win["llr"].astype(f).copy()
        for u in range(int(np.diff(cp).max())):
            has = np.diff(cp) > u
            post[has] = post[has] + c2v[cp[:-1][has] + u]
        x = post[col] - c2v
        v2c = np.where(x > clip, f(clip), np.where(x < -clip, f(-clip), x)).astype(f)
    return post


@pytest.mark.parametrize("T", [1, 2, 5])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3e38])
def test_posteriors(value, T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qbuild.build()
    from paper_2403_18901_gb300.learn import Wms
    dem = qdec.Dem(CODES["72"], 0.003, 6)
    params = preset("configured", k_guess=3)
    dec = qdec.Decoder(dem, params, max_shots=4)
    wms, win = Wms(dec, 1, T, 1), dem.window(3, 1, 1)
    rng = np.random.default_rng(T)
    w = rng.uniform(0.4, 0.9, size=(T, win["n_edges"])).astype(np.float32)
    w[rng.random(w.shape) < 0.005] = value
    synd = (rng.random((3, win["n_rows"])) < 0.2).astype(np.uint8)
    words = np.zeros((3, wms.rw * 32), np.uint8)
    words[:, :win["n_rows"]] = synd
    packed = np.packbits(words, axis=1, bitorder="little").view(np.int32)
    _, post = wms.loss(torch.from_numpy(w).cuda(), torch.from_numpy(packed).cuda(), want_post=True)
    with np.errstate(all="ignore"):
        for s in range(3):
            want = _posteriors(win, w, synd[s], params["clip"])
            got = post[s].cpu().numpy()
            assert np.array_equal(got, want, equal_nan=True), (np.nonzero(~((got == want) | np.isnan(got)))[0], s)
