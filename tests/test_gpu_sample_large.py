"""GPU test of the sampler on an experiment of many rounds: 1380 detector words, where
fewer than eight warps' detector rows and lists of fired columns fit a CTA.  Every
shot is compared with its definition: column c fires when word c mod 4 of
Philox4x32-10 (counter c / 4, shot, key seed) is below its threshold, and flips
its detectors and observables."""
import numpy as np
import pytest

from paper_2403_18901_gb300 import build as qbuild
from paper_2403_18901_gb300 import qdec
from paper_2403_18901_gb300.workloads import CODES

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _philox(ctr, key):
    """Philox4x32-10 of counters [n][4] (uint32) with one key."""
    c = [ctr[:, i].astype(np.uint64) for i in range(4)]
    k0, k1 = key
    low = np.uint64(0xFFFFFFFF)
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & low, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1),
             p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return np.stack(c, 1).astype(np.uint32)


def test_more_detectors_than_eight_rows_hold():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qbuild.build()
    dem = qdec.Dem(CODES["90"], 0.003, 980)
    assert dem.det_words == 1380
    seed, off, n = 0x1234567890AB, (1 << 33) - 3, 9
    det, obs = (x.cpu().numpy().view(np.uint32) for x in dem.sample(seed, off, n))
    cols = dem.columns()
    thr = np.floor(cols["prob"] * 4294967296.0 + 0.5).astype(np.uint32)
    groups = (dem.n_cols + 3) // 4
    for s in range(n):
        shot = off + s
        ctr = np.zeros((groups, 4), np.uint32)
        ctr[:, 0] = np.arange(groups)
        ctr[:, 1], ctr[:, 2] = shot & 0xFFFFFFFF, shot >> 32
        fired = np.nonzero(_philox(ctr, (seed & 0xFFFFFFFF, seed >> 32)).reshape(-1)[:dem.n_cols] < thr)[0]
        want = np.zeros(32 * dem.det_words, np.uint8)
        for c in fired:
            want[cols["col_dets"][cols["col_ptr"][c]:cols["col_ptr"][c + 1]]] ^= 1
        assert len(fired) > 500
        assert (np.unpackbits(det[s].view(np.uint8), bitorder="little") == want).all(), s
        assert obs[s] == np.bitwise_xor.reduce(cols["obs"][fired]), s
