"""The decoder's work as its users run it: what the performance of this repository is measured on.

Each case is one call (or one loop of calls) a program makes through the package's public classes:

* "pass"    -- a Monte-Carlo batch on device buffers, every sliding window decoded and committed (Decoder.decode_all);
* "host"    -- the same from host buffers to host buffers (Decoder.decode_host);
* "stream"  -- a real-time loop, one window after another for the few shots in flight (Decoder.decode_commit_static);
* "batch"   -- decoders of several codes and window sizes advanced together (Batch.step);
* "sample"  -- drawing detector shots from the error model (Dem.sample);
* "weights" -- the gradient of the learned min-sum weights over a batch of window samples (learn.Wms.grad);
* "ranker"  -- the gradient of the decimation ranker over a batch of candidate records (ranker.grad).

Codes, noise rates, rounds and decoder parameters are those of workloads.py, the tests and bench.py.
"""
import math

import numpy as np
import torch

from paper_2403_18901_gb300 import learn, qdec, ranker
from paper_2403_18901_gb300.workloads import CODES, preset


def listed():
    return [
        # the smallest call in use: one [[72,12,6]] shot decoded window by window as its rounds come in
        dict(name="stream_72_one_shot", kind="stream", code="72", rounds=6, p=0.003, preset="configured", k=3, shots=1),
        # the latency workload of the benchmark: one [[144,12,12]] shot in real time, 16 decision paths
        dict(name="stream_144_one_shot", kind="stream", code="144", rounds=12, p=0.003, preset="configured", k=4,
             shots=1),
        # a handful of shots with the paper's own decoder (22 paths), too few to fill the GPU
        dict(name="pass_144_paper_25", kind="pass", code="144", rounds=12, p=0.003, preset="paper", k=4, shots=25),
        # the headline workload: a Monte-Carlo batch of [[144,12,12]], (3,1) windows, 100 BP iterations, 16 paths
        dict(name="pass_144", kind="pass", code="144", rounds=12, p=0.003, preset="configured", k=4, shots=5000),
        # the paper's own decoder on a batch: short BP, most paths converge early
        dict(name="pass_144_paper", kind="pass", code="144", rounds=12, p=0.003, preset="paper", k=4, shots=9001),
        # the larger code at the low error rate, from and to host memory as an experiment's control program holds it
        dict(name="host_288", kind="host", code="288", rounds=18, p=0.002, preset="configured", k=4, shots=509),
        # decoding with learned per-edge weights in place of the normalisation factor
        dict(name="pass_144_weights", kind="pass", code="144", rounds=12, p=0.003, preset="configured", k=4, shots=2000,
             weights=25),
        # decoding with the learned decimation ranker
        dict(name="pass_144_ranker", kind="pass", code="144", rounds=12, p=0.003, preset="configured", k=4, shots=1201,
             ranker=True),
        # three codes with window sizes 2, 3 and 4 advanced together, the benchmark's batched uneven workload
        dict(name="batch_uneven", kind="batch", codes="90,108,144", Ws="2,3,4", p=0.003, preset="configured", k=4,
             shots=333),
        # shots for a logical error rate: the sampler alone
        dict(name="sample_144", kind="sample", code="144", rounds=12, p=0.003, shots=100000),
        # one training step's gradient of the learned weights, 25 unrolled iterations of an interior window
        dict(name="train_weights_144", kind="weights", code="144", rounds=12, p=0.003, T=25, ckpt=5, n=1024),
        # one training step's gradient of the ranker on the benchmark's minibatch
        dict(name="train_ranker", kind="ranker", n=65536),
    ]


# ---------------------------------------------------------------------------------------------------------------
# Cases of the same ranges.

_ROUNDS = {"72": 6, "90": 10, "108": 10, "144": 12, "288": 18}


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _us_per_window(code, W, pre, k):
    """Roughly what one window of one shot takes in a batch, for keeping drawn cases below the largest listed one."""
    c = CODES[code]
    us = (9.0 if pre == "configured" else 2.6) * (c["n"] / 144.0) ** 1.6 * (W / 3.0) ** 1.6 * (2 ** k / 16.0)
    return us * (1.6 if code == "288" else 1.0)


def draw(rng):
    kind = rng.choice(["pass", "pass", "pass", "host", "stream", "stream", "batch", "sample", "weights", "ranker"])
    if kind == "ranker":
        return dict(kind=kind, n=_log_int(rng, 1000, 200000))
    if kind == "batch":
        codes = rng.choice(["72,90", "90,108,144", "108,144", "72,144", "72,90,108"])
        return dict(kind=kind, codes=codes, Ws=rng.choice(["2,3", "2,3,4", "3"]), p=round(rng.uniform(0.001, 0.004), 5),
                    preset=rng.choice(["configured", "paper"]), k=rng.choice([3, 4]), shots=_log_int(rng, 11, 300))
    code = rng.choice(["72", "90", "108", "144", "144", "288"])
    rounds = rng.randint(max(4, _ROUNDS[code] // 2), _ROUNDS[code])
    p = round(rng.uniform(0.001, 0.004), 5)
    if kind == "sample":
        return dict(kind=kind, code=code, rounds=rounds, p=p, shots=_log_int(rng, 1000, 100000))
    if kind == "weights":
        code = rng.choice(["72", "90", "108", "144"])
        T = rng.randint(5, 25)
        return dict(kind=kind, code=code, rounds=_ROUNDS[code], p=p, T=T, ckpt=rng.randint(1, min(T, 7)),
                    n=_log_int(rng, 100, 1024))
    pre = rng.choice(["configured", "paper"])
    k = rng.choice([3, 4, 4, 5])
    case = dict(kind=kind, code=code, rounds=rounds, p=p, preset=pre, k=k)
    W = rng.choice([2, 3, 3, 3, 4])
    if code == "144" and pre == "paper" and rng.random() < 0.25:
        W, case["F"] = 5, 2
    if W != 3:
        case["W"] = W
    most = int(0.25e6 / (_us_per_window(code, W, pre, k) * max(1, rounds + 2 - W)))
    case["shots"] = rng.randint(1, 30) if kind == "stream" else _log_int(rng, 20, max(21, min(most, 9000)))
    if kind == "pass":
        what = rng.random()
        if what < 0.2:
            case["weights"] = rng.randint(10, 25)
        elif what < 0.4:
            case["ranker"] = True
        elif what < 0.55:
            case["reuse_msgs"] = 1
    return case


# ---------------------------------------------------------------------------------------------------------------
# What a program has in hand before the call.


def _params(case, W=None):
    over = dict(W=W if W is not None else case.get("W", 3), F=case.get("F", 1))
    if case.get("reuse_msgs"):
        over["reuse_msgs"] = 1
    if case.get("code") == "288":  # the larger code's deeper main branch and tree (bench.py, ranker section)
        over.update(d_max_main=40, d_max_other=case["k"] + 20)
        if case["preset"] == "paper":
            over.update(side_max=20, n_pre=16)
    return preset(case["preset"], case["k"], case["p"], **over)


def _weights(T, n_edges, gen):
    """Weights as training leaves them: scattered around the normalisation factor they start from."""
    w = 0.625 + 0.1 * torch.randn((T, n_edges), generator=gen)
    return w.clamp_(0.1, 1.2).cuda()


def _records(n, gen):
    """Candidate records as the decoder writes them: posteriors of the last four iterations on the 1/2 grid, their
    mean, unsatisfied neighbours, degree and block; labels are rare and go with negative posteriors."""
    centre = 6.0 + 9.0 * torch.randn((n, 1), generator=gen)
    h = (centre + 3.0 * torch.randn((n, 4), generator=gen)).clamp(-63.5, 63.5)
    x = torch.zeros((n, 8))
    x[:, 1:5] = torch.round(2.0 * h) / 2.0
    x[:, 0] = torch.round(2.0 * h.mean(1)) / 2.0
    x[:, 5] = torch.randint(0, 6, (n,), generator=gen).float()
    x[:, 6] = torch.randint(3, 7, (n,), generator=gen).float()
    x[:, 7] = torch.randint(0, 3, (n,), generator=gen).float()
    rec = torch.zeros((n, 12), dtype=torch.float32)
    rec[:, :8] = x
    ints = rec.view(torch.int32)
    ints[:, 8] = torch.arange(n, dtype=torch.int32) // 200
    ints[:, 9] = torch.randint(0, 2160, (n,), generator=gen).int()
    ints[:, 11] = (x[:, 0] <= 0.0).int()
    y = ((x[:, 0] <= 0.0) & (torch.rand(n, generator=gen) < 0.3)).to(torch.uint8)
    return rec.view(torch.uint8).cuda(), y.cuda()


def prepare(case, seed):
    gen = torch.Generator().manual_seed(int(seed))
    kind = case["kind"]
    if kind == "ranker":
        recs, labels = _records(case["n"], gen)
        return dict(case=case, params=ranker.init_params(int(seed) & 0xFFFF), recs=recs, labels=labels)
    if kind == "batch":
        members = []
        for code in case["codes"].split(","):
            dem = qdec.Dem(CODES[code], case["p"], _ROUNDS[code])
            for W in case["Ws"].split(","):
                n = case["shots"]
                dec = qdec.Decoder(dem, _params(dict(case, code=code), W=int(W)), max_shots=n)
                det, obs = dem.sample(seed, len(members) * n, n)
                members.append(dict(dem=dem, dec=dec, det=det, n=n))
        return dict(case=case, members=members, batch=qdec.Batch([m["dec"] for m in members]))
    dem = qdec.Dem(CODES[case["code"]], case["p"], case["rounds"])
    if kind == "sample":
        return dict(case=case, dem=dem, seed=int(seed))
    if kind == "weights":
        dec = qdec.Decoder(dem, preset("configured", 4, case["p"]), max_shots=1)
        wms = learn.Wms(dec, 1, T=case["T"], ckpt=case["ckpt"])
        return dict(case=case, dem=dem, dec=dec, wms=wms, synd=wms.sample(int(seed), 0, case["n"]),
                    w=_weights(wms.T, wms.n_edges, gen))
    n = case["shots"]
    dec = qdec.Decoder(dem, _params(case), max_shots=n)
    if case.get("weights"):
        for k in range(dec.n_windows):
            dec.set_weights(k, _weights(case["weights"], dec.window_info(k)["n_edges"], gen))
    if case.get("ranker"):
        dec.set_ranker(ranker.init_params(int(seed) & 0xFFFF).cpu().numpy())
    det, obs = dem.sample(int(seed), 0, n)
    state = dict(case=case, dem=dem, dec=dec, det=det, obs=obs)
    if kind == "host":
        state["det"] = det.cpu().numpy().view(np.uint32)
        state["obs"] = obs.cpu().numpy().view(np.uint32)
    return state


# ---------------------------------------------------------------------------------------------------------------
# One pass.


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ranker":
        n = case["n"]
        grad, loss = ranker.grad(state["params"], state["recs"], state["labels"], True, 10.0, 1.0 / n)
        return dict(grad=grad, loss=loss)
    if kind == "weights":
        grad, loss = state["wms"].grad(state["w"], state["synd"], 1.0 / case["n"])
        return dict(grad=grad, loss=loss)
    if kind == "sample":
        det, obs = state["dem"].sample(state["seed"], 0, case["shots"])
        return dict(det=det, obs=obs)
    if kind == "batch":
        members = state["members"]
        det = [m["det"].clone() for m in members]
        n = [m["n"] for m in members]
        pred = [torch.zeros(x, dtype=torch.int32, device="cuda") for x in n]
        resid = [torch.zeros(x, dtype=torch.int32, device="cuda") for x in n]
        for j in range(state["batch"].n_steps):
            state["batch"].step(j, det, n, pred, resid)
        return dict(det=det, pred=pred, resid=resid)
    dec, n = state["dec"], case["shots"]
    if kind == "host":
        pred, fail, n_fail = dec.decode_host(state["det"], state["obs"])
        return dict(pred=pred.view(np.int32), fail=fail.view(np.int32), n_fail=n_fail)
    det = state["det"].clone()
    if kind == "stream":
        pred = torch.zeros(n, dtype=torch.int32, device="cuda")
        resid = torch.zeros(n, dtype=torch.int32, device="cuda")
        for k in range(dec.n_windows):
            dec.decode_commit_static(k, det, n, pred, resid)
        return dict(det=det, pred=pred, resid=resid)
    pred = torch.empty(n, dtype=torch.int32, device="cuda")
    fail = torch.empty(n, dtype=torch.int32, device="cuda")
    n_fail = torch.zeros(1, dtype=torch.int64, device="cuda")
    dec.decode_all(det, state["obs"], n, pred, fail, n_fail)
    return dict(det=det, pred=pred, fail=fail, n_fail=n_fail)


# ---------------------------------------------------------------------------------------------------------------
# What a pass cannot do without.  Decoding: ten operations for one edge's share of one flooding iteration
# (Eq. (1)-(3): subtract, two compares of the clip, magnitude, two minimum compares, sign, scale, select, add).
# The number of edge iterations depends on the shots; these are typical counts per window at the listed sizes.


def _decode_work(case, code, rounds, W, F, shots):
    w = CODES[code]["n"] // 2
    windows = max(1, math.ceil((rounds + 1 - W) / F) + 1)
    edges = 30.7 * w * W  # edges of an interior window
    if case["preset"] == "configured":
        per_window = edges * 85 + 62.0 * w * W * (2 ** case["k"] * 12 + 20) * 10 * 0.04
    else:
        per_window = edges * 7 + 62.0 * w * W * (2 ** case["k"] * 4) * 6 * 0.016
    det_bytes = 4 * ((w * (rounds + 1) + 31) // 32)
    return shots * (2 * det_bytes + 12), 10.0 * shots * windows * per_window


def work(case):
    kind = case["kind"]
    if kind == "ranker":
        return dict(bytes=case["n"] * (32 + 1 + 4) + 2 * 641 * 4, flops=case["n"] * 6 * 64 * 9)
    if kind == "sample":
        w = CODES[case["code"]]["n"] // 2
        cols = w * (2 + 10 * case["rounds"])
        dets = w * (case["rounds"] + 1)
        return dict(bytes=case["shots"] * (4 * ((dets + 31) // 32) + 4), flops=case["shots"] * cols / 4 * 60)
    if kind == "weights":
        w = CODES[case["code"]]["n"] // 2
        edges = 30.7 * w * 3
        return dict(bytes=case["n"] * (4 * ((3 * w + 31) // 32) + 4) + 8 * edges * case["T"],
                    flops=case["n"] * edges * case["T"] * 30)
    if kind == "batch":
        b = f = 0
        for code in case["codes"].split(","):
            for W in case["Ws"].split(","):
                x, y = _decode_work(case, code, _ROUNDS[code], int(W), 1, case["shots"])
                b, f = b + x, f + y
        return dict(bytes=b, flops=f)
    b, f = _decode_work(case, case["code"], case["rounds"], case.get("W", 3), case.get("F", 1), case["shots"])
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------------------------------------------------------
# The computed numbers in 64 bits (decoding and sampling give whole numbers).


def _exact_ranker(s):
    p = s["params"].double()
    grid = lambda x, scale, lim: (x * scale).round().clamp(-lim, lim) / scale  # noqa: E731
    W1 = grid(p[:512], 64.0, 128.0).view(64, 8)
    b1 = grid(p[512:576], 128.0, 65536.0)
    W2 = grid(p[576:640], 64.0, 128.0)
    x = s["recs"].view(torch.float32)[:, :8].double()
    y = s["labels"].double()
    a = x @ W1.t() + b1
    h = a.clamp_min(0.0)
    z = h @ W2 + p[640]
    wy = torch.where(y > 0.5, 10.0, 1.0).double()
    loss = wy * (z.clamp_min(0.0) + torch.log1p(torch.exp(-z.abs())) - y * z)
    dz = wy * (torch.sigmoid(z) - y) / x.shape[0]
    dh = torch.where(a > 0.0, dz[:, None] * W2, torch.zeros_like(a))
    grad = torch.cat([(dh.t() @ x).reshape(-1), dh.sum(0), h.t() @ dz, dz.sum().reshape(1)])
    return dict(grad=grad, loss=loss)


def _exact_weights(case, s):
    """T unrolled iterations of weighted min-sum and the soft-syndrome loss, differentiated by torch."""
    win = s["dem"].window(3, 1, 1)
    nr, nc, ne, T = win["n_rows"], win["n_cols"], win["n_edges"], case["T"]
    col_of = np.repeat(np.arange(nc), np.diff(win["col_ptr"]))
    rows = [[] for _ in range(nr)]
    for e, j in enumerate(win["col_rows"]):
        rows[j].append(e)
    D = max(len(r) for r in rows)
    pad = np.full((nr, D), ne, np.int64)  # a check's edges, padded with the extra edge ne
    for j, r in enumerate(rows):
        pad[j, :len(r)] = r
    dev = "cuda"
    pad_t = torch.from_numpy(pad).to(dev)
    real = pad_t < ne
    col = torch.from_numpy(col_of).to(dev)
    llr = torch.from_numpy(win["llr"]).double().to(dev)
    back = torch.empty(ne, dtype=torch.int64, device=dev)  # edge -> its place in the padded rows
    flat = pad_t.reshape(-1)
    back[flat[flat < ne]] = torch.nonzero(flat < ne).reshape(-1)
    w = s["w"].double().requires_grad_(True)
    bits = s["synd"].long()
    j = torch.arange(nr, device=dev)
    synd = ((bits[:, j >> 5] >> (j & 31)) & 1).double()
    n, clip, eps = synd.shape[0], 50.0, 1e-7
    # the kernel clamps in 32 bits; the bound itself is part of the function
    lo, hi = float(np.float32(eps)), float(np.float32(1.0) - np.float32(eps))
    losses = []
    for a0 in range(0, n, 64):
        sy = synd[a0:a0 + 64]
        m = sy.shape[0]
        v = llr[col].expand(m, ne)
        for t in range(T):
            vp = torch.cat([v, torch.full((m, 1), float("inf"), dtype=v.dtype, device=dev)], 1)[:, flat].view(m, nr, D)
            with torch.no_grad():
                ap = vp.abs()
                i1 = ap.argmin(2, keepdim=True)
                i2 = ap.scatter(2, i1, float("inf")).argmin(2, keepdim=True)
                sgn = torch.where((vp < 0) & real, -1.0, 1.0).double()
                par = sgn.prod(2, keepdim=True) * (1.0 - 2.0 * sy[:, :, None])
                own = torch.arange(D, device=dev).view(1, 1, D) == i1
            m1 = vp.gather(2, i1) * sgn.gather(2, i1)
            m2 = vp.gather(2, i2) * sgn.gather(2, i2)
            c = (torch.where(own, m2, m1) * (sgn * par)).reshape(m, nr * D)[:, back] * w[t]
            post = llr.expand(m, nc).index_add(1, col, c)
            x = post[:, col] - c
            v = torch.where(x.abs() < clip, x, torch.where(x < 0, -clip, clip).double())
        th = torch.cat([torch.tanh(0.5 * post)[:, col], torch.ones((m, 1), dtype=v.dtype, device=dev)], 1)
        P = (0.5 * (1.0 - th[:, flat].view(m, nr, D).prod(2))).clamp(lo, hi)
        per = torch.where(sy > 0.5, -torch.log(P), -torch.log(1.0 - P)).mean(1)
        (per.sum() / n).backward()
        losses.append(per.detach())
    return dict(grad=w.grad, loss=torch.cat(losses))


def exact(case, seed):
    if case["kind"] == "ranker":
        return _exact_ranker(prepare(case, seed))
    if case["kind"] == "weights":
        return _exact_weights(case, prepare(case, seed))
    return None
