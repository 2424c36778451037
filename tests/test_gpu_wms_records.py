"""GPU test of the training kernel's kept check records: with more iterations than
its scratch keeps whole, every ckpt-th one's records are kept and the others
computed again.  One sample's gradient (no two additions to one place) and loss
are bit for bit those of a context that keeps every iteration, for spacings that
divide T and that do not, and a context's scratch follows ckpt."""
import numpy as np
import pytest

from paper_2403_18901_gb300 import build as qbuild
from paper_2403_18901_gb300 import qdec
from paper_2403_18901_gb300.workloads import CODES, preset

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def window():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qbuild.build()
    dem = qdec.Dem(CODES["72"], 0.003, 6)
    return dem, qdec.Decoder(dem, preset("configured", k_guess=3), max_shots=4)


def _scratch(dec, T, ckpt):
    from paper_2403_18901_gb300.learn import Wms
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    wms = Wms(dec, 1, T, ckpt)
    return wms, before - torch.cuda.mem_get_info()[0]


def test_gradients_do_not_depend_on_the_spacing(window):
    _, dec = window
    T, grads = 280, []
    for ckpt in (280, 1, 7, 16, 140, 279):
        wms, _ = _scratch(dec, T, ckpt)
        rng = np.random.default_rng(1)
        w = torch.from_numpy(rng.uniform(0.9, 1.2, size=(T, wms.n_edges)).astype(np.float32)).cuda()
        synd = wms.sample(77, 0, 4)
        out = [wms.grad(w, synd[i:i + 1].contiguous()) for i in range(4)]
        grads.append([(g.cpu(), l.cpu()) for g, l in out])
    assert sum(int((g[: T - 16] != 0).any()) for g, _ in grads[0]) > 0  # some flow past the last segment
    for got in grads[1:]:
        for (g, l), (g0, l0) in zip(got, grads[0]):
            assert torch.equal(g, g0) and torch.equal(l, l0)


def test_scratch_follows_the_spacing(window):
    _, dec = window
    wms, whole = _scratch(dec, 1000, 1000)
    del wms
    wms, spaced = _scratch(dec, 1000, 32)
    assert whole > 500 << 20 and spaced < whole / 8
