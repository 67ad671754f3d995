"""Timing cases of the Dion step: what a training loop asks of the library, through the binding's public calls.

A case is one call (or one short cycle of calls) on matrices in the state that training leaves them in:
parameters ~ N(0, 0.02^2), a momentum and a gradient that share a decaying low-rank signal under Gaussian noise,
and a right factor with unit-norm columns.  Calls used: ``Dion.step`` (standard and transposed form, fp32 and
bf16-operand mode), ``Dion.step_grouped``, ``Dion.lazy_step`` and the three ``Dion.dp_*`` calls.
"""
from __future__ import annotations

import math

import torch

from paper_2504_05295_b200 import binding

LR = 0.01
LAZY_EVERY = 4      # Lazy-Dion: one step that refreshes the right factor, then three that do not

# matrices of one transformer block, rows = out: (rows, columns, how many of this shape)
BLOCK_4096 = [(4096, 4096, 2), (1024, 4096, 2), (14336, 4096, 2), (4096, 14336, 1)]
BLOCK_768 = [(768, 768, 4), (3072, 768, 1), (768, 3072, 1)]


def listed():
    return [
        # the smallest matrix of the benchmark: latency of one call
        {"name": "step-256x512-r64", "kind": "step", "m": 256, "n": 512, "r": 64, "g": "f32", "mode": "fp32"},
        # an odd-sized parameter (vocabulary slices, fused heads): no dimension a multiple of 4
        {"name": "step-1001x333-r83", "kind": "step", "m": 1001, "n": 333, "r": 83, "g": "f32", "mode": "fp32"},
        # an ordinary hidden-size matrix at a low rank fraction
        {"name": "step-2048-r128", "kind": "step", "m": 2048, "n": 2048, "r": 128, "g": "f32", "mode": "fp32"},
        # full rank: the rule without compression (the panel is ill conditioned)
        {"name": "step-2048-full", "kind": "step", "m": 2048, "n": 2048, "r": 2048, "g": "f32", "mode": "fp32"},
        # the usual rank fraction 1/4 on one matrix of a large model
        {"name": "step-4096-r1024", "kind": "step", "m": 4096, "n": 4096, "r": 1024, "g": "f32", "mode": "fp32"},
        # bf16 gradients and bf16 operands (the reduced-precision mode)
        {"name": "bf16ops-8192-r512", "kind": "step", "m": 8192, "n": 8192, "r": 512, "g": "bf16", "mode": "bf16"},
        # a very large matrix at rank fraction 1/64: memory traffic counts
        {"name": "step-16384-r256", "kind": "step", "m": 16384, "n": 16384, "r": 256, "g": "f32", "mode": "fp32"},
        # transposed form on a tall feed-forward matrix: the panel sits on the short side
        {"name": "transposed-14336x4096-r1024", "kind": "transposed", "m": 14336, "n": 4096, "r": 1024, "g": "bf16",
         "mode": "fp32"},
        # compressed data-parallel sync: the three calls between which a rank all-reduces the factors
        {"name": "dp-4096x2048-r256", "kind": "dp", "m": 4096, "n": 2048, "r": 256, "g": "bf16", "mode": "fp32"},
        # Lazy-Dion, one refresh cycle
        {"name": "lazy-4096-r256", "kind": "lazy", "m": 4096, "n": 4096, "r": 256, "g": "f32", "mode": "fp32"},
        # every matrix of a small model (12 blocks of hidden size 768) in one call
        {"name": "grouped-768-12-blocks", "kind": "grouped", "block": 768, "layers": 12, "fraction": 0.25, "g": "bf16",
         "mode": "fp32"},
        # two blocks of the 4096-wide list (14 matrices) in one call: throughput
        {"name": "grouped-4096-2-blocks", "kind": "grouped", "block": 4096, "layers": 2, "fraction": 0.25, "g": "bf16",
         "mode": "fp32"},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    cap = 3.5e12      # floating-point operations: below those of the largest listed case
    while True:
        kind = rng.choice(["step", "step", "step", "step", "transposed", "dp", "lazy", "grouped"])
        mode = "bf16" if rng.random() < 0.15 else "fp32"
        g = rng.choice(["f32", "bf16"])
        if kind == "grouped":
            block = rng.choice([768, 768, 4096])
            case = {"kind": kind, "block": block, "layers": rng.randint(2, 12) if block == 768 else 1,
                    "fraction": rng.choice([0.0625, 0.125, 0.25]), "g": g, "mode": mode}
        else:
            m, n = _log_uniform(rng, 128, 16384), _log_uniform(rng, 128, 16384)
            fraction = rng.choice([1 / 64, 1 / 16, 1 / 8, 1 / 4, 1 / 4, 1.0])
            if kind == "lazy":
                fraction = min(fraction, 0.25)
            shape = rng.random()
            if shape < 0.6:      # most parameters have dimensions in multiples of 64
                m, n = max(128, m // 64 * 64), max(128, n // 64 * 64)
            elif shape < 0.8:
                m, n = m // 4 * 4, n // 4 * 4
            r = max(1, int(fraction * min(m, n)))
            if (fraction == 1.0 and min(m, n) > 3072) or m * n > 1.5e8:
                continue
            if shape >= 0.6 and 8.0 * m * n * r > 1e11:      # odd sizes of this weight are rare
                continue
            case = {"kind": kind, "m": m, "n": n, "r": r, "g": g, "mode": mode}
        if work(case)["flops"] <= cap:
            return case


# ---- inputs ------------------------------------------------------------------------------------------------------

def _classes(case):
    """(rows, columns, rank, count) of the shapes that a case steps."""
    if case["kind"] != "grouped":
        return [(case["m"], case["n"], case["r"], 1)]
    block = BLOCK_768 if case["block"] == 768 else BLOCK_4096
    return [(m, n, max(1, int(case["fraction"] * min(m, n))), k * case["layers"]) for m, n, k in block]


def _full_rank(case):
    return any(2 * r > min(m, n) for m, n, r, _ in _classes(case))


_CONTEXTS = {}


def _context(mode):
    """One library context per precision, kept like a training program keeps its optimizer."""
    if mode not in _CONTEXTS:
        precision = binding.PREC_BF16_OPERANDS if mode == "bf16" else binding.PREC_FP32
        _CONTEXTS[mode] = binding.Dion(precision=precision)
    return _CONTEXTS[mode]


def _stack(count, rows, cols, dtype):
    """`count` dense matrices in one buffer, each on a 256-byte boundary, and a view of each."""
    pitch = (rows * cols + 127) // 128 * 128
    flat = torch.zeros(count, pitch, dtype=dtype, device="cuda")
    return flat, [flat[k, :rows * cols].view(rows, cols) for k in range(count)]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))

    def randn(rows, cols):
        return torch.randn((rows, cols), generator=gen, device="cuda", dtype=torch.float32)

    g_dtype = torch.bfloat16 if case["g"] == "bf16" else torch.float32
    transposed = case["kind"] == "transposed"
    mats, buffers = [], []
    for m, n, r, count in _classes(case):
        q_rows = m if transposed else n
        Xf, Xs = _stack(count, m, n, torch.float32)
        Mf, Ms = _stack(count, m, n, torch.float32)
        _, Gs = _stack(count, m, n, g_dtype)
        Qf, Qs = _stack(count, q_rows, r, torch.float32)
        df = torch.zeros(count, (r + 31) // 32 * 32, device="cuda")
        for k in range(count):
            # signal of decaying strength (Gaussian factors are orthonormal to 1/sqrt(rows)) shared by gradient and
            # momentum; the momentum has averaged some noise away
            ks = min(64, m, n)
            us, vs = randn(m, ks) / math.sqrt(m), randn(n, ks) / math.sqrt(n)
            us *= torch.pow(2.0, -0.5 * torch.arange(ks, dtype=torch.float32, device="cuda"))
            Xs[k].copy_(randn(m, n).mul_(0.02))
            Ms[k].copy_(randn(m, n).mul_(0.3).addmm_(us, vs.t(), alpha=5.0))
            Gs[k].copy_(randn(m, n).mul_(0.1).addmm_(us, vs.t()))
            q = randn(q_rows, r)
            if 2 * r > min(m, n):      # past its first steps a full-rank run has a nearly orthonormal right factor
                q = torch.linalg.qr(q)[0]
            Qs[k].copy_(q / torch.linalg.vector_norm(q, dim=0))
            mats.append((Xs[k], Ms[k], Gs[k], Qs[k], df[k, :r]))
        buffers.append((Xf, Mf, Qf, df))
    state = {"kind": case["kind"], "opt": _context(case["mode"]), "mats": mats, "buffers": buffers}
    if case["kind"] == "dp":
        m, n, r = case["m"], case["n"], case["r"]
        state["P"], state["W"] = torch.zeros(m, r, device="cuda"), torch.zeros(n, r, device="cuda")
        state["flag"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    return state


def run(state):
    opt, kind = state["opt"], state["kind"]
    if kind == "grouped":
        opt.step_grouped(state["mats"], LR)
        return state["buffers"]
    X, M, G, Q, d = state["mats"][0]
    if kind == "lazy":
        for t in range(LAZY_EVERY):
            opt.lazy_step(X, M, G, Q, LR, refresh=(t == 0), colnorm_out=d)
    elif kind == "dp":
        desc = binding.matrix_desc(X, M, G, Q, d)
        opt.dp_project(desc, state["P"], state["flag"])
        opt.dp_factor(desc, state["P"], state["W"], state["flag"])
        opt.dp_finish(desc, state["P"], state["W"], state["flag"], LR)
        return state["buffers"], state["P"], state["W"]
    else:
        opt.step(X, M, G, Q, LR, colnorm_out=d, transposed=(kind == "transposed"))
    return state["buffers"]


# ---- what a pass cannot do without -------------------------------------------------------------------------------

def work(case):
    """X, M, Q read and written once, G read once; the four rank-r products and one Cholesky QR of the panel
    (Gram matrix and triangular solve at rows r^2 each, r^3 / 3)."""
    g_bytes = 2 if case["g"] == "bf16" else 4
    nbytes = flops = 0.0
    for m, n, r, count in _classes(case):
        q_rows = m if case["kind"] == "transposed" else n
        panel_rows = n if case["kind"] in ("transposed", "lazy") else m
        orth = 2.0 * panel_rows * r * r + r ** 3 / 3.0
        state = 16.0 * m * n + g_bytes * m * n + 8.0 * q_rows * r
        if case["kind"] == "lazy":      # a refresh is two more products and the orthonormalization
            nbytes += count * LAZY_EVERY * state
            flops += count * (LAZY_EVERY * 6.0 * m * n * r + 4.0 * m * n * r + orth)
        else:
            # the factors that the data-parallel calls hand out are outputs (and inputs of the next call) too
            nbytes += count * (state + (16.0 * (m + n) * r if case["kind"] == "dp" else 0.0))
            flops += count * (8.0 * m * n * r + orth)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["mode"] == "bf16":      # operands rounded to 8 bits
        return {"rel": 1e-2, "max": 0.3}
    if _full_rank(case):
        # the thin-QR factor of a square panel follows its condition number (1e4 and more): Q moves by 1e-3 when P is
        # merely formed by another 32-bit product
        return {"rel": 1e-2, "max": 0.3}
    return {"rel": 1e-4}      # the library's stated bound in its fp32 mode
