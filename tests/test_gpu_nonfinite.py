"""GPU test of messages that are not finite: learned weights of infinity, NaN
or near the largest float on some edges, and no clip at all (clip = infinity)
with checks of one active column (no peeling at the start), whose message is
the clip.  inf - inf makes an edge's input NaN: like an infinite one it is never
the smallest nor the second smallest of its check.  Bit-exact against the
oracle, whose comparisons leave a NaN out the same way.

The weights are compared over the BP on the full window (its outcome, its
iterations, the correction or the columns it ranks first), where every check has
several finite inputs beside a NaN; each edge is infinite for one iteration, so
that the posteriors that rank the columns are numbers."""
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


@pytest.mark.parametrize("mode", [1, 2, 3])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3e38])
def test_weights_that_are_not_finite(value, mode):
    n, k = 64, 1
    o = oracle_dem("72", 0.003, 6)
    params = preset("configured", k_guess=3)
    rng = np.random.default_rng(9)
    win = o.window(3, 1, k)
    w = rng.uniform(0.45, 0.9, size=(12, win["n_edges"])).astype(np.float32)
    for t in range(1, 6):
        w[t, rng.choice(win["n_edges"], 6, replace=False)] = value
    dec = qdec.Decoder(qdec.Dem(CODES["72"], 0.003, 6), params, max_shots=n)
    dec.set_launch(mode)
    dec.set_weights(k, torch.from_numpy(w).cuda())
    det, _ = o.sample(61, 0, n)
    corr = torch.zeros((n, dec.corr_words), dtype=torch.int32, device="cuda")
    trace = torch.zeros((n, dec.trace_bytes), dtype=torch.uint8, device="cuda")
    dec.decode_window(k, torch.from_numpy(det.view(np.int32)).cuda(), n, corr, None, trace)
    bits = np.unpackbits(det.view(np.uint8), axis=1, bitorder="little")
    got = np.unpackbits(corr.cpu().numpy().view(np.uint8), axis=1, bitorder="little")[:, :win["n_cols"]]
    traces, row0, ended = trace.cpu().numpy(), win["r0"] * o.w, [0, 0]
    for s in range(n):
        want, info, otr = o.decode_window(params, k, bits[s, row0:row0 + win["n_rows"]].copy(), trace=True,
                                          weights={k: w})
        tr = dec.parse_trace(traces[s])
        assert (tr["head"][0], tr["head"][3]) == (int(info["prebp_converged"]), info["prebp_iters"]), s
        ended[int(info["prebp_converged"])] += 1
        if info["prebp_converged"]:
            assert (got[s] == np.asarray(want)[:win["n_cols"]]).all(), s
        else:
            assert (tr["short_cols"][:info["n_short"]] == otr["short_cols"]).all(), s
    assert min(ended) > 0


@pytest.mark.parametrize("mode", [1, 2])
def test_no_clip(mode):
    params = dict(preset("configured", k_guess=3), clip=float("inf"), peel_at_init=0)
    _pipeline("72", 6, 0.003, params, n=48, seed=62, trace_windows=(0, 1, 2, 3, 4), mode=mode)
