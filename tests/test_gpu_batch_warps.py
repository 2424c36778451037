"""GPU test of batched steps in CTAs of few warps with a path schedule: 16 and 32
decision paths (so that paths queue for the warps, resume from snapshots and are
preempted), CTAs of one to eight warps, more shots than resident CTAs, so that
every CTA starts shots after others.  Bit-exact against the per-decoder path,
itself bit-exact to the oracle."""
import pytest

from paper_2403_18901_gb300 import build as qbuild
from paper_2403_18901_gb300 import qdec
from paper_2403_18901_gb300.workloads import CODES, preset

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MEMBERS = [("72", 6, 3, 5, 400), ("72", 6, 2, 4, 500)]  # (code, rounds, W, k_guess, shots)


@pytest.fixture(scope="module")
def members():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    qbuild.build()
    qdec.lib()
    out = []
    for i, (key, R, W, k, n) in enumerate(MEMBERS):
        dem = qdec.Dem(CODES[key], 0.004, R)
        dec = qdec.Decoder(dem, preset("configured", k_guess=k, p=0.004, W=W), max_shots=n)
        det0, _ = dem.sample(seed=410 + i, shot_offset=0, n_shots=n)
        det, pred, resid = det0.clone(), *(torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
        corr = torch.zeros((n, dec.corr_words), dtype=torch.int32, device="cuda")
        for j in range(dec.n_windows):
            dec.decode_window(j, det, n, corr)
            dec.commit(j, corr, n, det, pred, resid)
        torch.cuda.synchronize()
        out.append(dict(dec=dec, n=n, det0=det0, ref=[t.cpu() for t in (det, pred, resid)]))
    return out


@pytest.mark.parametrize("warps,ctas", [(1, 2), (2, 2), (3, 1), (4, 2), (8, 2)])
def test_scheduled_paths_in_small_ctas(members, warps, ctas):
    b = qdec.Batch([m["dec"] for m in members])
    n = [m["n"] for m in members]
    det = [m["det0"].clone() for m in members]
    pred, resid = ([torch.zeros(x, dtype=torch.int32, device="cuda") for x in n] for _ in range(2))
    for j in range(b.n_steps):
        b.set_shape(j, warps, ctas)
        assert b.info(j)["warps"] == warps and sum(n) > b.info(j)["ctas_per_sm"] * 152
        b.step(j, det, n, pred, resid)
    torch.cuda.synchronize()
    for m, *got in zip(members, det, pred, resid):
        assert all(torch.equal(x, y.cpu()) for x, y in zip(m["ref"], got))
