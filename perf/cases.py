"""The timed cases of the library: what a program that uses it does per call.

A case is a dict of plain values; ``prepare`` makes what such a program holds
before the call (device inputs, the plan with its filters set, output
buffers it keeps), ``run`` makes one pass through the public entry points,
``work`` counts the bytes and operations of the pass that cannot be left out
(each input read once, each output written once; conventional FFT operation
counts), and ``exact`` gives the same outputs in 64 bits from plain torch.
Inputs are the synthetic ones of the parity tests: signals uniform in
[-1, 1], Gaussian filter taps (optionally Hann-windowed), unit L2 norm.
"""
import math

import torch

from paper_1910_01972_gb300 import BatchPlan, Plan, ols_conv
from paper_1910_01972_gb300 import _native

BATCH_M = (33, 65, 129, 257, 513, 1025)
FLAGS = {"convolve": _native.OLS_FLAG_FP32, "power": _native.OLS_FLAG_FP32, "derivative": _native.OLS_FLAG_FP32,
         "real": _native.OLS_FLAG_R2R, "fp16split": _native.OLS_FLAG_TC_FP16SPLIT,
         "bf16split": _native.OLS_FLAG_TC_BF16SPLIT}


def listed():
    return [
        # one signal, one filter: the smallest call in use, where latency and the host path count
        {"name": "single_filter", "kind": "convolve", "Ns": 65536, "F": 1, "M": 64, "N": 512, "window": False,
         "keep_out": True},
        # a block of a live stream through a filter bank, into a buffer the program keeps; ragged length
        {"name": "stream_block", "kind": "convolve", "Ns": 65521, "F": 32, "M": 257, "N": 2048, "window": True,
         "keep_out": True},
        # the filter bank of the benchmark: a recorded signal, 32 Hann-windowed filters
        {"name": "filter_bank", "kind": "convolve", "Ns": 1 << 23, "F": 32, "M": 257, "N": 2048, "window": True,
         "keep_out": False},
        # long filters at the segment length the plan picks by itself (8192); odd length
        {"name": "long_filters", "kind": "convolve", "Ns": (1 << 22) + 1, "F": 24, "M": 1025, "N": 0, "window": False,
         "keep_out": False},
        # short filters at the plan's own segment length (256); odd length
        {"name": "short_filters", "kind": "convolve", "Ns": 3000017, "F": 32, "M": 33, "N": 0, "window": False,
         "keep_out": False},
        # many signals of uneven length with banks of their own, one persistent launch
        {"name": "uneven_batch", "kind": "batch", "B": 16, "lo_log2": 16, "hi_log2": 21, "F_lo": 8, "F_hi": 128,
         "shapes": 3},
        # a training step of learnable filters: forward, gradients of the signal and of the filters
        {"name": "train_step", "kind": "train", "Ns": 1 << 22, "F": 16, "M": 129, "N": 1024},
        # the same on a short excerpt with a small bank, segment length left to the library
        {"name": "train_small", "kind": "train", "Ns": 20011, "F": 8, "M": 65, "N": 0},
        # real signal, real filters
        {"name": "real_bank", "kind": "real", "Ns": 1 << 23, "F": 32, "M": 257, "N": 2048, "window": True,
         "keep_out": False},
        # power of the filtered signal (the detection chain's input), longer filters
        {"name": "power_bank", "kind": "power", "Ns": 2500003, "F": 32, "M": 513, "N": 4096, "window": True,
         "keep_out": False},
        # derivative of the filtered signal
        {"name": "derivative_bank", "kind": "derivative", "Ns": 1 << 22, "F": 16, "M": 129, "N": 1024,
         "window": False, "keep_out": False},
        # the split-precision form on the tensor cores
        {"name": "split_bank", "kind": "fp16split", "Ns": 1 << 22, "F": 64, "M": 512, "N": 4096, "window": False,
         "keep_out": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["convolve", "convolve", "convolve", "train", "train", "batch", "real", "power", "derivative",
                       "fp16split", "bf16split"])
    if kind == "batch":
        return {"kind": kind, "B": rng.randint(4, 24), "lo_log2": 15, "hi_log2": rng.choice([18, 19, 20]), "F_lo": 8,
                "F_hi": rng.choice([32, 64, 128]), "shapes": rng.randrange(1 << 20)}
    F = _log(rng, 1, 64)
    M = _log(rng, 16, 1500)
    # segment length: the plan's own choice, or one a program names (room for the overlaps of the adjoint)
    N = 0
    if rng.random() < 0.4:
        N = min(8192, max(256, 1 << ((2 * M - 1).bit_length() + rng.randint(0, 2))))
    Ns = _log(rng, 1 << 13, min(1 << 23, (1 << 28) // F))
    if kind == "train":
        Ns = min(Ns, (1 << 26) // F)
        return {"kind": kind, "Ns": Ns, "F": F, "M": M, "N": N}
    return {"kind": kind, "Ns": Ns, "F": F, "M": M, "N": N, "window": rng.random() < 0.5,
            "keep_out": rng.random() < 0.5}


def _shapes(case):
    """(Ns, F, M) of every problem of a batch, from the case alone."""
    import random
    r = random.Random(case["shapes"])
    out = []
    for _ in range(case["B"]):
        n = int(round(2.0 ** r.uniform(case["lo_log2"], case["hi_log2"])))
        out.append((n, r.randint(case["F_lo"], case["F_hi"]), r.choice(BATCH_M)))
    return out


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _signal(g, n, real=False):
    x = torch.rand(n if real else 2 * n, generator=g, device="cuda").mul_(2.0).sub_(1.0)
    return x if real else torch.view_as_complex(x.view(n, 2))


def _filters(g, F, M, window, real=False):
    h = torch.randn((F, M) if real else (F, M, 2), generator=g, device="cuda", dtype=torch.float64)
    h = h if real else torch.view_as_complex(h)
    if window and M > 2:
        h = h * torch.hann_window(M, periodic=False, device="cuda", dtype=torch.float64)
    h = h / torch.linalg.vector_norm(h, dim=1, keepdim=True)
    return h.to(torch.float32 if real else torch.complex64).contiguous()


def _inputs(case, seed):
    g = _gen(seed)
    if case["kind"] == "batch":
        sh = _shapes(case)
        return [_signal(g, n) for n, _, _ in sh], [_filters(g, f, m, False) for _, f, m in sh]
    real = case["kind"] == "real"
    s = _signal(g, case["Ns"], real)
    h = _filters(g, case["F"], case["M"], case.get("window", False), real)
    if case["kind"] != "train":
        return s, h
    n = case["Ns"] - case["M"] + 1
    gy = torch.view_as_complex(torch.randn((case["F"], n, 2), generator=g, device="cuda"))
    return s, h, gy


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        ss, hs = _inputs(case, seed)
        sh = _shapes(case)
        plan = BatchPlan([x[0] for x in sh], [x[2] for x in sh], [x[1] for x in sh], model_only=True)
        plan.set_filters(hs)
        return {"kind": kind, "plan": plan, "s": ss, "out": plan.outputs()}
    if kind == "train":
        s, h, gy = _inputs(case, seed)
        return {"kind": kind, "s": s.requires_grad_(), "h": h.requires_grad_(), "gy": gy, "N": case["N"]}
    s, h = _inputs(case, seed)
    plan = Plan(case["M"], case["F"], case["N"], FLAGS[kind])
    (plan.set_filters_real if kind == "real" else plan.set_filters)(h)
    out = None
    if case["keep_out"]:
        out = torch.empty((case["F"], case["Ns"] - case["M"] + 1), device="cuda",
                          dtype=torch.float32 if kind in ("real", "power") else torch.complex64)
    return {"kind": kind, "plan": plan, "s": s, "out": out}


def run(state):
    kind = state["kind"]
    if kind == "batch":
        return state["plan"].convolve(state["s"], state["out"])
    if kind == "train":
        y = ols_conv(state["s"], state["h"], state["N"])
        ds, dh = torch.autograd.grad(y, (state["s"], state["h"]), state["gy"])
        return {"y": y.detach(), "ds": ds, "dh": dh}
    plan, s, out = state["plan"], state["s"], state["out"]
    if kind == "real":
        return plan.convolve_real(s, out)
    if kind == "power":
        return plan.convolve_power(s, out)
    if kind == "derivative":
        return plan.convolve_derivative(s, out)
    return plan.convolve(s, out)


def _segment(M):
    """The shortest segment length with at most a quarter of it discarded (for the operation count only)."""
    return min(8192, max(256, 1 << (4 * M - 1).bit_length()))


def _one(Ns, F, M, N):
    """(segments, complex FFTs, operations) of one overlap-and-save pass."""
    N = N or _segment(M)
    nseg = -(-(Ns - M + 1) // (N - M + 1))
    return nseg * ((F + 1) * 5.0 * N * math.log2(N) + F * 6.0 * N)


def work(case):
    if case["kind"] == "batch":
        w = {"bytes": 0.0, "flops": 0.0}
        for n, f, m in _shapes(case):
            w["bytes"] += 8.0 * (n + f * m + f * (n - m + 1))
            w["flops"] += _one(n, f, m, 0)
        return w
    Ns, F, M, N = case["Ns"], case["F"], case["M"], case["N"]
    nout, flops = Ns - M + 1, _one(Ns, F, M, N)
    if case["kind"] == "train":
        # forward: s, h in, y out; backward: s, h, gy in, ds, dh out
        return {"bytes": 8.0 * (3 * Ns + 3 * F * M + 2 * F * nout), "flops": 2 * flops}
    if case["kind"] == "real":
        return {"bytes": 4.0 * (Ns + F * M + F * nout), "flops": flops / 2}
    out = 4.0 if case["kind"] == "power" else 8.0
    return {"bytes": 8.0 * (Ns + F * M) + out * F * nout, "flops": flops}


def _conv64(s, h):
    """Valid convolution of s with every row of h in complex128."""
    n, m = s.shape[0], h.shape[1]
    p = 1 << (n - 1).bit_length()
    S = torch.fft.fft(s.to(torch.complex128), p)
    y = torch.empty((h.shape[0], n - m + 1), dtype=torch.complex128, device=s.device)
    for f in range(h.shape[0]):
        y[f] = torch.fft.ifft(S * torch.fft.fft(h[f].to(torch.complex128), p))[m - 1:n]
    return y


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        ss, hs = _inputs(case, seed)
        return [_conv64(s, h) for s, h in zip(ss, hs)]
    if kind == "train":
        s, h, gy = _inputs(case, seed)
        n, m = s.shape[0], h.shape[1]
        p = 1 << (n - 1).bit_length()
        Sc = torch.fft.fft(s.to(torch.complex128), p).conj()
        ds = torch.zeros(p, dtype=torch.complex128, device=s.device)
        dh = torch.empty(h.shape, dtype=torch.complex128, device=s.device)
        for f in range(h.shape[0]):
            G = torch.fft.fft(gy[f].to(torch.complex128), p)
            ds += G * torch.fft.fft(h[f].to(torch.complex128).conj().resolve_conj().flip(0), p)
            c = torch.fft.ifft(G * Sc)               # c[l] = sum_j g[j] conj(s[j - l]), l = k - (m - 1)
            dh[f] = torch.cat([c[p - (m - 1):], c[:1]])
        return {"y": _conv64(s, h), "ds": torch.fft.ifft(ds)[:n].contiguous(), "dh": dh}
    s, h = _inputs(case, seed)
    y = _conv64(s, h)
    if kind == "real":
        return y.real.contiguous()
    if kind == "power":
        return y.real.square() + y.imag.square()
    if kind == "derivative":
        d = torch.empty_like(y)
        d[:, 1:-1] = (y[:, 2:] - y[:, :-2]) / 2
        d[:, 0], d[:, -1] = y[:, 1] - y[:, 0], y[:, -1] - y[:, -2]
        return d
    return y
