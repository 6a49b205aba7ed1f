"""The work a user of the channeliser has it do, as timed cases.

Each case is one call (or one training step) through the public entry points:
``ppf.Plan`` for single streams and batches of streams, its ``backward`` for
the adjoint, ``autograd.PolyphaseFilterBank`` for a step of tap fitting and
``beams.BeamSet`` for many uneven beams in one launch.  ``listed`` names the
cases, ``draw`` gives more of the same ranges, ``prepare`` makes inputs, plan
and buffers, ``run`` makes one pass, ``work`` counts what a pass cannot do
without and ``exact`` gives the result in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1511_03599_gb300 import autograd, beams, ppf

CHANNELS = (32, 64, 128, 256, 384, 512, 768, 1024, 1536, 2048, 3072, 4096)
BEAM_CHANNELS = (64, 128, 256, 512, 1024, 2048, 4096)
IN_BYTES = {"ci8": 2, "ci16": 4, "cf32": 8}
OUT_BYTES = {"c64": 8, "c16": 4}
SIGMA = {"ci8": 16.0, "ci16": 2000.0, "cf32": 1.0}
MAX_SAMPLES = 1 << 27          # of a drawn case
EXACT_BYTES = 1 << 34          # 64-bit results are computed up to this much work


def listed():
    return [
        # a block of a live stream, handed over as it arrives: 64 spectra of the benchmark's channel count
        {"name": "block_c512_t8_ci8", "kind": "forward", "C": 512, "T": 8, "S": 64, "streams": 1, "in": "ci8", "out": "c64"},
        # the plain PFB of the first workload: 4096 spectra of complex floats, a call of ordinary size
        {"name": "plain_c256_t8_cf32", "kind": "forward", "C": 256, "T": 8, "S": 4096, "streams": 1, "in": "cf32", "out": "c64"},
        # the benchmark's workload: a long recording of 8-bit samples
        {"name": "long_c512_t8_ci8", "kind": "forward", "C": 512, "T": 8, "S": 1 << 19, "streams": 1, "in": "ci8", "out": "c64"},
        # the tap / precision sweep: 16-bit samples, 16 taps, half-precision spectra
        {"name": "sweep_c512_t16_ci16_c16", "kind": "forward", "C": 512, "T": 16, "S": 1 << 17, "streams": 1, "in": "ci16", "out": "c16"},
        # the same sweep's long filters, on floats; a ragged count
        {"name": "taps_c512_t64_cf32", "kind": "forward", "C": 512, "T": 64, "S": 50021, "streams": 1, "in": "cf32", "out": "c64"},
        # fine channels from 8-bit samples, the benchmark's largest channel count
        {"name": "fine_c4096_t8_ci8", "kind": "forward", "C": 4096, "T": 8, "S": 30011, "streams": 1, "in": "ci8", "out": "c64"},
        # a channel count that is no power of two (the paper's example is 3072), on 16-bit samples
        {"name": "fine_c3072_t8_ci16", "kind": "forward", "C": 3072, "T": 8, "S": 12289, "streams": 1, "in": "ci16", "out": "c64"},
        # several antennas at once: independent streams of floats in one launch
        {"name": "streams_c1024_t4_cf32", "kind": "forward", "C": 1024, "T": 4, "S": 3001, "streams": 12, "in": "cf32", "out": "c64"},
        # a step of tap fitting, forward and both gradients, at the differentiable workload's shape
        {"name": "train_c256_t16", "kind": "train", "C": 256, "T": 16, "S": 4096, "streams": 64, "in": "cf32", "out": "c64"},
        # the adjoint at the benchmark's shape, 8-bit input
        {"name": "adjoint_c512_t8_ci8", "kind": "adjoint", "C": 512, "T": 8, "S": 1 << 17, "streams": 1, "in": "ci8", "out": "c64"},
        # the adjoint with the sweep's 32 taps
        {"name": "adjoint_c512_t32_ci8", "kind": "adjoint", "C": 512, "T": 32, "S": 1 << 16, "streams": 1, "in": "ci8", "out": "c64"},
        # many receivers' sub-bands: uneven beams in one persistent launch
        {"name": "beams_24", "kind": "beams", "beams": 24, "S_min": 1 << 10, "S_max": 1 << 15, "shapes": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("forward",) * 7 + ("train", "adjoint", "adjoint", "beams"))
    if kind == "beams":
        lo = _log_int(rng, 64, 1024)
        return {"kind": kind, "beams": rng.randint(6, 24), "S_min": lo, "S_max": lo * rng.randint(4, 16),
                "shapes": rng.randrange(1 << 30)}
    C = rng.choice(CHANNELS)
    T = rng.choice((rng.randint(1, 8), 8, rng.randint(9, 16), 16, rng.randint(17, 64)))
    if kind == "train":
        C, T, dtype = min(C, 1024), min(T, 16), "cf32"
    else:
        dtype = rng.choice(("ci8", "ci8", "ci16", "cf32"))
    out = rng.choice(("c64", "c64", "c16")) if kind == "forward" else "c64"
    samples = _log_int(rng, 1 << 15, MAX_SAMPLES if kind == "forward" else MAX_SAMPLES // 2)
    streams = rng.choice((1, 1, 1, rng.randint(2, 16), rng.randint(17, 64)))
    if kind == "train":
        streams = max(2, streams)
    while streams > 1 and samples // (C * streams) < 4:
        streams //= 2
    return {"kind": kind, "C": C, "T": T, "S": max(3, samples // (C * streams)), "streams": streams, "in": dtype, "out": out}


# ------------------------------------------------------------------ inputs
def _taps(C, T, scale=1.0):
    n = np.arange(C * T, dtype=np.float64)
    w = 0.54 - 0.46 * np.cos(2.0 * np.pi * n / (C * T - 1))
    return (np.sinc((n - (C * T - 1) / 2.0) / C) * w * scale).astype(np.float32)


def _noise(shape, dtype, gen):
    """Gaussian samples of the type, interleaved (re, im) along the last axis."""
    z = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    if dtype == "cf32":
        return z
    lim = 127 if dtype == "ci8" else 32767
    return z.mul_(SIGMA[dtype]).round_().clamp_(-lim, lim).to(torch.int8 if dtype == "ci8" else torch.int16)


def _beam_shapes(case):
    rng = np.random.default_rng(case["shapes"])
    n = case["beams"]
    C = [int(c) for c in rng.choice(BEAM_CHANNELS, n)]
    T = [int(t) for t in rng.choice([4, 8, 16], n)]
    S = [int(s) for s in rng.integers(case["S_min"], case["S_max"] + 1, n)]
    return C, T, S


def _tap_scale(case):
    return 1.0 / math.sqrt(case["C"]) if case["out"] == "c16" else 1.0   # keeps half-precision spectra in range


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    if case["kind"] == "beams":
        return [_noise((c * (s + t - 1), 2), "ci8", gen) for c, t, s in zip(*_beam_shapes(case))]
    C, T, S, ns = case["C"], case["T"], case["S"], case["streams"]
    lead = (ns,) if ns > 1 else ()
    x = _noise(lead + (C * (S + T - 1), 2), case["in"], gen)
    if case["kind"] == "forward":
        return [x]
    g = torch.randn(lead + (S, C), dtype=torch.complex64, device="cuda", generator=gen)
    if case["kind"] == "train":
        x = torch.view_as_complex(x)
    return [x, g]


def prepare(case, seed):
    ins = _inputs(case, seed)
    state = {"kind": case["kind"], "ins": ins}
    if case["kind"] == "beams":
        C, T, S = _beam_shapes(case)
        state["set"] = beams.BeamSet(C, T, S, [_taps(c, t) for c, t in zip(C, T)])
        state["outs"] = [torch.empty((s, c), dtype=torch.complex64, device="cuda") for c, s in zip(C, S)]
        state["set"].bind(ins, state["outs"])
        return state
    h = _taps(case["C"], case["T"], _tap_scale(case))
    if case["kind"] == "train":
        state["bank"] = autograd.PolyphaseFilterBank(case["C"], case["T"], h).cuda()
        state["bank"].plan()
        ins[0].requires_grad_(True)
        return state
    state["plan"] = ppf.Plan(case["C"], case["T"], h, case["in"], case["out"])
    state["streams"] = case["streams"] if case["streams"] > 1 else None
    if case["kind"] == "forward":
        state["out"] = state["plan"].empty_output(case["S"], device="cuda", n_streams=state["streams"])
    return state


def run(state):
    kind, ins = state["kind"], state["ins"]
    if kind == "beams":
        state["set"].execute()
        return state["outs"]
    if kind == "forward":
        return state["plan"].execute(ins[0], out=state["out"], n_streams=state["streams"])
    if kind == "adjoint":
        return list(state["plan"].backward(ins[1], ins[0]))
    y = state["bank"](ins[0])
    gx, gh = torch.autograd.grad(y, (ins[0], state["bank"].taps), ins[1])
    return [y.detach(), gx, gh]


# -------------------------------------------------------------------- work
def _flops(C, T):
    return 2 * (2 * T - 1) + 5 * math.log2(C)       # a sample's FIR and radix-2 transform


def work(case):
    if case["kind"] == "beams":
        shapes = list(zip(*_beam_shapes(case)))
        return {"bytes": sum(2 * c * (s + t - 1) + 8 * c * s + 4 * c * t for c, t, s in shapes),
                "flops": sum(c * s * _flops(c, t) for c, t, s in shapes)}
    C, T, S, ns = case["C"], case["T"], case["S"], case["streams"]
    raw, out, taps = ns * C * (S + T - 1), ns * C * S, 4 * C * T
    forward = raw * IN_BYTES[case["in"]] + out * OUT_BYTES[case["out"]] + taps
    adjoint = out * 8 + raw * (IN_BYTES[case["in"]] + 8) + 2 * taps    # G and x read, both gradients written
    f, a = out * _flops(C, T), out * (8 * T + 5 * math.log2(C))        # both sums of the adjoint: 4 T each
    if case["kind"] == "forward":
        return {"bytes": forward, "flops": f}
    if case["kind"] == "adjoint":
        return {"bytes": adjoint, "flops": a}
    return {"bytes": forward + adjoint, "flops": f + a}


# ------------------------------------------------------------------- exact
def _fir64(x, h, S):
    """x: (raw rows, C) complex128, h: (T, C) float64."""
    y = torch.zeros((S, x.shape[1]), dtype=torch.complex128, device=x.device)
    for t in range(h.shape[0]):
        y += h[t] * x[t:t + S]
    return y


def _forward64(x, h, C, T):
    """One stream of interleaved samples -> its spectra, in 64 bits, in pieces of rows."""
    rows = x.reshape(-1, C, 2)
    S = rows.shape[0] - T + 1
    h = torch.from_numpy(h.astype(np.float64)).to(x.device).reshape(T, C)
    out = torch.empty((S, C), dtype=torch.complex128, device=x.device)
    step = max(1, (1 << 24) // C)
    for lo in range(0, S, step):
        n = min(step, S - lo)
        z = torch.view_as_complex(rows[lo:lo + n + T - 1].double())
        out[lo:lo + n] = torch.fft.fft(_fir64(z, h, n), dim=-1)
    return out


def _adjoint64(x, g, h, C, T):
    """One stream: gradients with respect to its samples and to the taps, in 64 bits."""
    rows = x.reshape(-1, C, 2)
    S = rows.shape[0] - T + 1
    h = torch.from_numpy(h.astype(np.float64)).to(x.device).reshape(T, C)
    gx = torch.zeros((S + T - 1, C), dtype=torch.complex128, device=x.device)
    gh = torch.zeros((T, C), dtype=torch.float64, device=x.device)
    step = max(1, (1 << 24) // C)
    for lo in range(0, S, step):
        n = min(step, S - lo)
        gy = torch.fft.ifft(g.reshape(S, C)[lo:lo + n].to(torch.complex128), dim=-1, norm="forward")
        z = torch.view_as_complex(rows[lo:lo + n + T - 1].double())
        for t in range(T):
            gx[lo + t:lo + t + n] += h[t] * gy
            gh[t] += (gy.real * z[t:t + n].real + gy.imag * z[t:t + n].imag).sum(dim=0)
    return gx, gh


def _half_pairs(y):
    return torch.view_as_real(y)


def exact(case, seed):
    if work(case)["bytes"] > EXACT_BYTES:
        return None
    ins = _inputs(case, seed)
    if case["kind"] == "beams":
        C, T, S = _beam_shapes(case)
        return [_forward64(x, _taps(c, t), c, t) for x, c, t in zip(ins, C, T)]
    C, T, ns = case["C"], case["T"], case["streams"]
    h = _taps(C, T, _tap_scale(case))
    xs = torch.view_as_real(ins[0]) if ins[0].is_complex() else ins[0]
    xs = list(xs) if ns > 1 else [xs]
    pack = (lambda v: torch.stack(v)) if ns > 1 else (lambda v: v[0])
    y = None
    if case["kind"] != "adjoint":
        y = pack([_forward64(x, h, C, T) for x in xs])
        if case["kind"] == "forward":
            return _half_pairs(y) if case["out"] == "c16" else y
    gs = list(ins[1]) if ns > 1 else [ins[1]]
    pairs = [_adjoint64(x, g, h, C, T) for x, g in zip(xs, gs)]
    gx = pack([p[0].reshape(-1) for p in pairs])
    gh = sum(p[1] for p in pairs).reshape(-1)
    return [gx, gh] if case["kind"] == "adjoint" else [y, gx, gh]
