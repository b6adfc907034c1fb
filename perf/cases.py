"""Workloads of the channel estimator, through the calls a receiver's program makes.

A case is a plain dict: "kind" says which call, the rest are its sizes and options.

    estimate   received blocks on the GPU -> channel estimate (pk.estimate)
    train      relaxed pilot tanh(theta): loss, gradients of the blocks and of theta
    adjoint    a real-valued pilot: forward and both adjoint halves, called directly
    host       received blocks in page-locked host memory -> estimate in host memory
    serve      a burst of uneven requests through the native serving loop

Received blocks follow the multiplexed-pilot model: K transmitters at cyclic shifts of one
m-sequence, complex Gaussian taps with an exponential power-delay profile (0.3 per tap,
unit power per link), white noise at the case's SNR, complex64.
"""
import math

import numpy as np
import torch

import paper_2206_05506_gb300 as pk
from paper_2206_05506_gb300 import serve
from paper_2206_05506_gb300.autograd import relaxed_estimate

# characteristic polynomials x^r + sum x^t + 1 (primitive), exponents t below r
TAPS = {5: (2,), 6: (1,), 7: (1,), 8: (4, 3, 2), 9: (4,), 10: (3,), 11: (2,),
        12: (6, 4, 1), 13: (4, 3, 1)}
ROWS = 4096            # rows handled at once while inputs or 64-bit results are made


def listed():
    return [
        # one small frame: launch and call latency
        {"name": "frame_small_fp32", "kind": "estimate", "r": 7, "F": 1, "M": 8, "K": 2,
         "L": 16, "dtype": "fp32", "cp": 0, "rule": "kl", "snr": 10.0},
        # the paper's scale, 128 frames a call: plain FP32 and TF32
        {"name": "paper_fp32", "kind": "estimate", "r": 10, "F": 128, "M": 64, "K": 8,
         "L": 64, "dtype": "fp32", "cp": 0, "rule": "kl", "snr": 10.0},
        {"name": "paper_tf32", "kind": "estimate", "r": 10, "F": 128, "M": 64, "K": 8,
         "L": 64, "dtype": "tf32", "cp": 0, "rule": "kl", "snr": 10.0},
        # the large batch of long pilots: reduced precision, and plain FP32
        {"name": "bulk_fp16", "kind": "estimate", "r": 12, "F": 512, "M": 128, "K": 16,
         "L": 128, "dtype": "fp16", "cp": 0, "rule": "kl", "snr": 10.0},
        {"name": "bulk_e4m3", "kind": "estimate", "r": 12, "F": 256, "M": 128, "K": 16,
         "L": 128, "dtype": "e4m3", "cp": 0, "rule": "kl", "snr": 0.0},
        {"name": "bulk_fp32", "kind": "estimate", "r": 12, "F": 512, "M": 128, "K": 16,
         "L": 128, "dtype": "fp32", "cp": 0, "rule": "kl", "snr": 20.0},
        # few lags (short channels, a sounding of one transmitter), the library's choice
        {"name": "few_lags_auto", "kind": "estimate", "r": 12, "F": 256, "M": 128, "K": 1,
         "L": 16, "dtype": "auto", "cp": 0, "rule": "kl", "snr": 10.0},
        # rows with the cyclic prefix still in front, shifts spread evenly over the pilot
        {"name": "spread_cp_bf16", "kind": "estimate", "r": 11, "F": 128, "M": 37, "K": 4,
         "L": 128, "dtype": "bf16", "cp": 128, "rule": "spread", "snr": 10.0},
        # one step of pilot optimisation
        {"name": "train_step", "kind": "train", "N": 1023, "F": 64, "M": 64, "K": 8, "L": 64,
         "snr": 10.0},
        # a short real-valued pilot of composite length, in a layer of a larger receiver
        {"name": "adjoint_ragged", "kind": "adjoint", "N": 300, "F": 16, "M": 40, "K": 3,
         "L": 100, "snr": 10.0},
        # one 64-antenna frame of 16 slots from host memory: the frame latency
        {"name": "host_frame_fp16", "kind": "host", "r": 11, "F": 16, "M": 64, "K": 4,
         "L": 128, "dtype": "fp16", "snr": 10.0},
        # uneven requests that arrive together, on the plain FP32 path
        {"name": "serve_fp32", "kind": "serve", "requests": 48, "dtype": "fp32", "mix": 1,
         "snr": 10.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["estimate"] * 5 + ["train", "adjoint", "host", "serve", "serve"])
    snr = float(rng.choice([0, 10, 20, 30]))
    if kind == "serve":
        return {"kind": kind, "requests": _log(rng, 4, 96), "mix": rng.randrange(1 << 20),
                "dtype": rng.choice(["fp16", "fp32"]), "snr": snr}
    if kind in ("train", "adjoint"):
        N = rng.choice([(1 << rng.randint(6, 11)) - 1, _log(rng, 60, 2100)])
        M, K = _log(rng, 2, 64), rng.randint(1, 16)
        L = _log(rng, 1, max(1, min(128, N // K)))
        F = _log(rng, 1, max(1, min(64, (1 << 22) // (N * M))))
        return {"kind": kind, "N": N, "F": F, "M": M, "K": K, "L": L, "snr": snr}
    r = rng.randint(7, 12)
    N = (1 << r) - 1
    K = rng.randint(1, 16)
    rule = "spread" if kind == "estimate" and rng.random() < 0.25 else "kl"
    L = _log(rng, 1, min(256, N // K))
    M = rng.choice([_log(rng, 1, 256), 16, 32, 64, 128])
    most = (1 << 25) if kind == "host" else (1 << 28)          # received samples a call
    F = _log(rng, 1, max(1, min(512, most // (N * M), (1 << 39) // (N * M * K * L))))
    case = {"kind": kind, "r": r, "F": F, "M": M, "K": K, "L": L, "snr": snr,
            "dtype": rng.choice(["fp32", "fp32", "fp16", "bf16", "e4m3", "tf32", "auto"])}
    if kind == "estimate":
        case["cp"] = L if rng.random() < 0.25 else 0
        case["rule"] = rule
    return case


def _mseq(r):
    a = np.zeros((1 << r) - 1 + r, dtype=np.uint8)
    a[0] = 1
    for t in range((1 << r) - 1):
        a[t + r] = (a[t] + sum(int(a[t + i]) for i in TAPS[r])) & 1
    return a[:(1 << r) - 1].copy()


def _shifts(c, N):
    step = c["L"] if c.get("rule", "kl") == "kl" else N // c["K"]
    k, l = np.arange(c["K"])[:, None], np.arange(c["L"])[None, :]
    return torch.from_numpy((k * step + l).reshape(-1)).cuda()


def _gauss(gen, *shape):
    return torch.randn(*shape, dtype=torch.complex64, device="cuda", generator=gen)


def _blocks(gen, pilot, F, M, K, L, lags, snr, cp=0):
    """(received blocks [F, M, cp + N], channels [F, M, K, L])"""
    N, A = pilot.numel(), F * M
    w = torch.exp(-0.3 * torch.arange(L, device="cuda", dtype=torch.float64))
    amp = torch.sqrt(w / w.sum()).to(torch.float32)
    S = torch.fft.fft(pilot.to(torch.complex64))
    Y = torch.empty((A, cp + N), dtype=torch.complex64, device="cuda")
    h = torch.empty((A, K, L), dtype=torch.complex64, device="cuda")
    for a in range(0, A, ROWS):
        n = min(ROWS, A - a)
        h[a:a + n] = _gauss(gen, n, K, L) * amp
        x = torch.zeros((n, N), dtype=torch.complex64, device="cuda")
        x[:, lags] = h[a:a + n].reshape(n, K * L)
        y = torch.fft.ifft(torch.fft.fft(x) * S)
        Y[a:a + n, cp:] = y + _gauss(gen, n, N) * 10.0 ** (-snr / 20)
    if cp:
        Y[:, :cp] = Y[:, N:]
    return Y.view(F, M, cp + N), h.view(F, M, K, L)


def _gen(seed):
    return torch.Generator("cuda").manual_seed(int(seed))


# the request mix of a busy cell
MIX_M, MIX_R, MIX_L = (32, 64, 128, 256), (8, 9, 10, 11), (16, 32, 64)


def _mix(c):
    rng = np.random.default_rng(c["mix"])
    out = []
    for _ in range(c["requests"]):
        M, r, L = (int(rng.choice(v)) for v in (MIX_M, MIX_R, MIX_L))
        K = int(rng.integers(1, min(((1 << r) - 1) // L, 16) + 1))
        out.append((M, r, K, L))
    return out


def _bits_of(N):
    return _mseq(N.bit_length())


def _serve_inputs(c, seed):
    """(requests' shapes, one page-locked block per request)"""
    gen, shapes, ys = _gen(seed), _mix(c), []
    for M, r, K, L in shapes:
        bits = _mseq(r)
        p = torch.from_numpy(1.0 - 2.0 * bits).to("cuda", torch.float32)
        lags = torch.arange(K * L, device="cuda")
        ys.append(_blocks(gen, p, 1, M, K, L, lags, c["snr"])[0][0].cpu().pin_memory())
    return shapes, ys


def _inputs(c, seed):
    gen = _gen(seed)
    if c["kind"] in ("train", "adjoint"):
        N = c["N"]
        theta = torch.randn(N, device="cuda", generator=gen)
        p = torch.tanh(theta)
        Y, h = _blocks(gen, p, c["F"], c["M"], c["K"], c["L"], _shifts(c, N), c["snr"])
        G = _gauss(gen, c["F"], c["M"], c["K"], c["L"])
        return {"Y": Y, "h": h, "theta": theta, "p": p, "G": G}
    bits = _mseq(c["r"])
    p = torch.from_numpy(1.0 - 2.0 * bits).to("cuda", torch.float32)
    Y, h = _blocks(gen, p, c["F"], c["M"], c["K"], c["L"], _shifts(c, bits.size), c["snr"],
                   c.get("cp", 0))
    return {"Y": Y, "bits": bits, "p": p}


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "serve":
        shapes, ys = _serve_inputs(c, seed)
        out = torch.zeros(sum(M * K * L for M, _, K, L in shapes), dtype=torch.complex64).pin_memory()
        srv = serve.NativeServer(_bits_of, dtype=c["dtype"], slots=4, max_batch_rows=256)
        srv.prepare(sorted({(1 << r) - 1 for _, r, _, _ in shapes}), caps=serve.CAPACITIES[:2])
        reqs, off = [], 0
        for i, ((M, r, K, L), y) in enumerate(zip(shapes, ys)):
            reqs.append(serve.Request(i, 0.0, M, (1 << r) - 1, K, L, y.data_ptr(),
                                      out.data_ptr() + 8 * off))
            off += M * K * L
        return {"c": c, "srv": srv, "reqs": reqs, "ys": ys, "out": out}
    s = _inputs(c, seed)
    s["c"] = c
    if c["kind"] == "train":
        s["Y"].requires_grad_(True)
        s["theta"].requires_grad_(True)
    elif c["kind"] != "adjoint":
        s["pilot"] = pk.Pilot(s["bits"])
        if c["kind"] == "host":
            s["Y"] = s["Y"].cpu().pin_memory()
            s["out"] = torch.zeros((c["F"], c["M"], c["K"], c["L"]), dtype=torch.complex64).pin_memory()
    return s


def run(s):
    c = s["c"]
    if c["kind"] == "estimate":
        return pk.estimate(s["Y"], s["pilot"], c["K"], c["L"], dtype=c["dtype"],
                           cp_len=c["cp"], shift_rule=c["rule"])
    if c["kind"] == "train":
        H = relaxed_estimate(s["Y"], s["theta"], c["K"], c["L"])
        loss = (H - s["h"]).abs().pow(2).mean()
        dY, dtheta = torch.autograd.grad(loss, (s["Y"], s["theta"]))
        return {"H": H.detach(), "loss": loss.detach(), "dY": dY, "dtheta": dtheta}
    if c["kind"] == "adjoint":
        H = pk.estimate_real_pilot(s["Y"], s["p"], c["K"], c["L"])
        dY, dp = pk.backward(s["p"], s["Y"], s["G"], c["K"], c["L"])
        return {"H": H, "dY": dY, "dp": dp}
    if c["kind"] == "host":
        return pk.estimate_host(s["Y"], s["pilot"], c["K"], c["L"], dtype=c["dtype"],
                                out=s["out"])
    s["srv"].run(s["reqs"])
    return s["out"]


def work(case):
    c = case
    if c["kind"] == "serve":
        b = f = 0
        for M, r, K, L in _mix(c):
            b += 8 * M * ((1 << r) - 1 + K * L)
            f += 2 * M * r << r
        return {"bytes": b, "flops": f}
    A, KL = c["F"] * c["M"], c["K"] * c["L"]
    if c["kind"] in ("train", "adjoint"):
        N = c["N"]
        # forward: Y -> H; backward: G, Y -> dY; the true channels of the loss
        b = 8 * A * (3 * N + 2 * KL) + (8 * A * KL if c["kind"] == "train" else 0) + 12 * N
        return {"bytes": b, "flops": 3 * A * 5 * 2 * N * math.log2(2 * N)}
    N = (1 << c["r"]) - 1
    # a fast transform over the pilot's shift group: r levels of complex additions
    return {"bytes": 8 * A * (N + KL), "flops": 2 * A * c["r"] << c["r"]}


def _correlate(Y, p, lags):
    """(1/N) sum_n Y[.., n] p[(n - j) mod N] in 64 bits, for the given lags"""
    N, A = p.numel(), Y.shape[0]
    P = torch.fft.fft(p.to(torch.complex128)).conj()
    H = torch.empty((A, lags.numel()), dtype=torch.complex128, device="cuda")
    for a in range(0, A, ROWS):
        y = Y[a:a + ROWS].to("cuda", torch.complex128)
        H[a:a + ROWS] = torch.fft.ifft(torch.fft.fft(y) * P)[:, lags] / N
    return H


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "serve":
        shapes, ys = _serve_inputs(c, seed)
        out = []
        for (M, r, K, L), y in zip(shapes, ys):
            p = torch.from_numpy(1.0 - 2.0 * _mseq(r)).cuda()
            out.append(_correlate(y, p, torch.arange(K * L, device="cuda")).reshape(-1))
        return torch.cat(out)
    s = _inputs(c, seed)
    F, M, K, L = c["F"], c["M"], c["K"], c["L"]
    if c["kind"] not in ("train", "adjoint"):
        N = s["bits"].size
        Y = s["Y"].view(F * M, -1)[:, c.get("cp", 0):]
        return _correlate(Y, s["p"].double(), _shifts(c, N)).view(F, M, K, L)
    N, KL = c["N"], K * L
    p = torch.tanh(s["theta"].double()) if c["kind"] == "train" else s["p"].double()
    H = _correlate(s["Y"].view(F * M, N), p, torch.arange(KL, device="cuda")).view(F, M, K, L)
    if c["kind"] == "train":
        e = H - s["h"].to(torch.complex128)
        loss = e.abs().pow(2).mean()
        G = 2 * e / e.numel()
    else:
        G = s["G"].to(torch.complex128)
    Gf = torch.zeros((F * M, N), dtype=torch.complex128, device="cuda")
    Gf[:, :KL] = G.view(F * M, KL)
    Gf = torch.fft.fft(Gf)
    dY = torch.fft.ifft(Gf * torch.fft.fft(p.to(torch.complex128))) / N
    cross = (Gf.conj() * torch.fft.fft(s["Y"].view(F * M, N).to(torch.complex128))).sum(0)
    dp = torch.fft.ifft(cross).real / N
    if c["kind"] == "train":
        return {"H": H, "loss": loss, "dY": dY.view(F, M, N), "dtheta": dp * (1 - p * p)}
    return {"H": H, "dY": dY.view(F, M, N), "dp": dp}
