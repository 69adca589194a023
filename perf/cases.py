"""Optimizer steps as a training program makes them: which ones, their inputs and their tolerances.

A case is one optimizer step through the public entry points of `binding.py`:

  kind "single"   one matrix, `orthdion_step`
  kind "noalloc"  one small matrix, `orthdion_step_noalloc` (built-in scratch)
  kind "group"    every matrix of a Llama-style model, `orthdion_step_grouped`
  kind "shard"    the local phases of one rank of a column-sharded matrix, `orthdion_shard_phase`

Ranges (`listed` and `draw` alike): matrices from 128 x 128 to 14336 x 4096, ranks from 1 to 1024 (16 up
to a quarter of the smaller side where the tensor engine runs), whole models of up to about 1.75
billion parameters, both normalisations, float32 and bfloat16 weights and gradients, both forms of the
error feedback, decay on and off, sizes that are multiples of nothing.
"""
import math

import numpy as np
import torch

from paper_2605_16341_b200 import binding as od

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
MODES = {"orth": od.MODE_ORTH, "dion": od.MODE_COLNORM}
ETA = 0.01
MOST_ELEMENTS = 1_750_000_000     # of a model: the largest listed one


def _single(name, m, n, r, mode="orth", x="bf16", g="bf16", kind="single", beta=0.0, wd=0.0, diag=0):
    return dict(name=name, kind=kind, m=m, n=n, r=r, mode=mode, x=x, g=g, beta=beta, wd=wd, diag=diag)


def _group(name, layers, d, dkv, dff, r, mode="orth", x="bf16", g="bf16", beta=0.0, wd=0.0, diag=0):
    return dict(name=name, kind="group", layers=layers, d=d, dkv=dkv, dff=dff, r=r, mode=mode, x=x, g=g,
                beta=beta, wd=wd, diag=diag)


def listed():
    return [
        # the smallest layers of a model in full precision: one small matrix, latency only
        _single("tiny_256x512_r16_f32", 256, 512, 16, x="f32", g="f32"),
        # a hook that may not allocate steps one small layer with the built-in scratch
        _single("noalloc_520x384_r64", 520, 384, 64, kind="noalloc"),
        # sizes that fit no tile (odd width, rank that is no multiple of 16): the fp32 engine
        _single("ragged_1023x777_r40_f32", 1023, 777, 40, x="f32", g="f32"),
        # one attention projection at rank d/16
        _single("attn_4096x4096_r256", 4096, 4096, 256),
        # one MLP projection at both ends of the rank sweep: little rank and Dion's normalisation,
        # bound by memory; the largest rank, bound by the factorisations
        _single("mlp_11008x4096_r32_dion", 11008, 4096, 32, mode="dion"),
        _single("mlp_11008x4096_r1024", 11008, 4096, 1024),
        # one rank's share (of four) of a column-sharded 4096 x 14336 down projection
        _single("shard_4096x3584_r512", 4096, 3584, 512, kind="shard"),
        # the 320M model of the paper (width 768, MLP 2048, rank fraction 1/4), its residual form of the
        # error feedback and its weight decay
        _group("model_320m_beta", 24, 768, 768, 2048, 192, beta=0.95, wd=0.1),
        # float32 weights under bfloat16 gradients, odd widths, the diagnostics that an adaptive rank reads
        _group("mixed_1000_r272_diag", 4, 1000, 376, 2712, 272, x="f32", diag=1),
        # every matrix of a 1.1B model, both normalisations (the second at rank d/16)
        _group("model_1b_r512", 22, 2048, 2048, 5632, 512),
        _group("model_1b_r128_dion", 22, 2048, 2048, 5632, 128, mode="dion"),
        # one of four pipeline stages of an 8B model
        _group("stage_8b_r512", 8, 4096, 1024, 14336, 512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rank(rng, small):
    """A rank that the tensor engine takes: a 64th up to a quarter of the smaller side, from 16 to 1024."""
    top = max(16, min(small // 4, 1024))
    return max(16, min(_log(rng, max(16, top // 16), top + 8) // 16 * 16, top // 16 * 16))


def draw(rng):
    kind = rng.choices(["small", "ragged", "matrix", "shard", "group"], [2, 1, 3, 1, 4])[0]
    mode = rng.choices(["orth", "dion"], [2, 1])[0]
    x, g = rng.choices([("bf16", "bf16"), ("f32", "f32"), ("f32", "bf16")], [4, 1, 1])[0]
    beta, wd = rng.choices([(0.0, 0.0), (0.0, 0.1), (0.95, 0.1)], [4, 1, 1])[0]
    diag = rng.choices([0, 1], [7, 1])[0]
    if kind == "ragged":          # the fp32 engine: any size, any rank
        m, n = _log(rng, 64, 1400), _log(rng, 64, 1400)
        r = max(1, min(_log(rng, 1, 96), m // 2, n // 2))
        if r % 16 == 0:
            r -= 1
        c = _single("", m, n, r, mode, x, g, beta=beta, wd=wd, diag=diag)
    elif kind == "small":
        m, n = _log(rng, 128, 1024), _log(rng, 128, 1024) // 8 * 8
        c = _single("", m, n, _rank(rng, min(m, n)), mode, x, g, kind=rng.choice(["single", "noalloc"]), beta=beta, wd=wd)
    elif kind == "matrix":
        m, n = _log(rng, 1024, 14336), _log(rng, 1024, 8192) // 8 * 8
        c = _single("", m, n, _rank(rng, min(m, n)), mode, x, g, beta=beta, wd=wd, diag=diag)
    elif kind == "shard":
        m, n = _log(rng, 1024, 8192), _log(rng, 1024, 8192) // 8 * 8
        c = _single("", m, n, _rank(rng, min(m, n)), mode, x, g, kind="shard", beta=beta, wd=wd)
    else:
        d = _log(rng, 512, 4096) // 8 * 8
        if rng.random() < 0.6:    # most models have round widths
            d = max(512, d // 128 * 128)
        dkv = rng.choice([d, max(128, d // 4 // 8 * 8)])
        dff = int(d * rng.uniform(2.6, 3.5)) // 8 * 8
        most = max(1, min(32, MOST_ELEMENTS // (2 * d * d + 2 * d * dkv + 3 * d * dff)))
        r = min(_rank(rng, min(d, dkv)), 512)
        c = _group("", _log(rng, 1, most), d, dkv, dff, r, mode, x, g, beta, wd, diag)
    del c["name"]
    return c


def _shapes(case):
    """(m, n) -> how many such matrices, in the model's order of first appearance."""
    if case["kind"] != "group":
        return {(case["m"], case["n"]): 1}
    d, dkv, dff = case["d"], case["dkv"], case["dff"]
    out = {}
    for s in [(d, d), (dkv, d), (dkv, d), (d, d), (dff, d), (dff, d), (d, dff)]:
        out[s] = out.get(s, 0) + case["layers"]
    return out


def _orthonormal(count, rows, cols, gen, first=None):
    """Batch of rows x cols matrices with random orthonormal columns (two Cholesky passes over N(0,1)
    columns), the leading ones `first` where that is given."""
    a = torch.randn(count, rows, cols, generator=gen, device="cuda") / math.sqrt(rows)
    if first is not None:
        a[:, :, :first.shape[2]] = first
    for _ in range(2):
        chol = torch.linalg.cholesky(a.mT @ a)
        a = torch.linalg.solve_triangular(chol, a.mT, upper=False).mT
    return a.contiguous()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    r = case["r"]
    xdt, gdt = DTYPES[case["x"]], DTYPES[case["g"]]
    hs, X, M, G, Q = [], [], [], [], []     # a plan per matrix; the matrices of a shape in one tensor
    for (m, n), count in _shapes(case).items():
        h = od.orthdion_create(m, n, r, 0.95, ETA, case["wd"], MODES[case["mode"]])
        od.orthdion_set_dtypes(h, xdt, gdt)
        if case["beta"]:
            od.orthdion_set_ef(h, case["beta"], case["beta"])
        if case["diag"]:
            od.orthdion_set_diagnostics(h, case["diag"])
        hs += [h] * count
        # Gradients as in pre-training: noise under a few dominant directions (singular values from ten
        # times the noise's largest down to five times).  The buffer of a run under way holds
        # several such gradients, and the right factor of the last step has found the directions.
        k = min(64, r)
        s = (math.sqrt(m) + math.sqrt(n)) / math.sqrt(n) * torch.linspace(10.0, 5.0, k, device="cuda")
        U, V = _orthonormal(count, m, k, gen), _orthonormal(count, n, k, gen)
        Q.append(_orthonormal(count, n, r, gen, first=V))
        X.append(torch.empty(count, m, n, dtype=xdt, device="cuda"))
        M.append(torch.empty(count, m, n, device="cuda"))
        G.append(torch.empty(count, m, n, dtype=gdt, device="cuda"))
        for i in range(count):
            spike = (U[i] * s) @ V[i].T
            noise = torch.randn(m, n, generator=gen, device="cuda")
            G[-1][i] = spike + noise / math.sqrt(n)
            noise.normal_(generator=gen)
            M[-1][i] = 3.0 * spike + noise * (3.0 / math.sqrt(n))
            noise.normal_(generator=gen)
            X[-1][i] = 0.02 * noise
    state = dict(kind=case["kind"], hs=hs, X=X, M=M, G=G, Q=Q, diag=case["diag"])
    if case["kind"] == "noalloc":
        state["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    else:
        state["ws"] = od.alloc_workspace(od.orthdion_workspace_bytes_grouped(hs))
    if case["kind"] == "group":
        each = [[t for stack in part for t in stack] for part in (X, M, G, Q)]
        state["table"] = od.PointerTable(hs, *each)
    else:
        state["one"] = [part[0][0] for part in (X, M, G, Q)]
    if case["kind"] == "shard":
        state["phases"] = 4 if case["mode"] == "orth" else 3
    return state


def run(state):
    kind, hs = state["kind"], state["hs"]
    out = {"X": state["X"], "M": state["M"], "Q": state["Q"]}
    if kind == "group":
        od.orthdion_step_grouped(state["table"], state["ws"])
    elif kind == "noalloc":
        od.orthdion_step_noalloc(hs[0], *state["one"], state["status"])
        out["status"] = state["status"]
    elif kind == "shard":
        # (between two phases the ranks sum a small buffer; that exchange is not the framework's)
        for phase in range(state["phases"]):
            od.orthdion_shard_phase(hs[0], phase, *state["one"], state["ws"])
    else:
        od.orthdion_step(hs[0], *state["one"], state["ws"])
    if state["diag"]:
        # what an adaptive rank reads after every step (all but the count of iterations)
        recs = od.orthdion_last_diagnostics(hs, state["ws"])
        out["diag"] = np.array([[rec[k] for k in od.DIAG_NAMES[:-1]] for rec in recs])
    return out


def work(case):
    size = {"bf16": 2, "f32": 4}
    r, orth = case["r"], case["mode"] == "orth"
    nbytes = flops = 0
    for (m, n), count in _shapes(case).items():
        nbytes += count * (m * n * (2 * size[case["x"]] + size[case["g"]] + 8) + 8 * n * r)
        flops += count * (8 * m * n * r + 6 * (m + (n if orth else 0)) * r * r + 2 * (2 if orth else 1) * r ** 3 // 3)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # About four times what one step differs from the same step in float64.  Tensor engine: two products
    # in a row from two-term bf16 splits (2^-16 each) behind a factorisation, up to 5e-5 in Q (largest
    # entry 3e-4).  bfloat16 weights are one spacing off where a value lies at a boundary: 4e-4, 8e-3.
    # The fp32 engine (odd widths, ranks that are no multiple of 16): 3e-6, 2.5e-5.
    if case["x"] == "bf16":
        return {"rel": 1.5e-3, "max": 0.032}
    if case["kind"] == "single" and (case["r"] % 16 or case["n"] % 8):
        return {"rel": 1.2e-5, "max": 1e-4}
    return {"rel": 2e-4, "max": 1.2e-3}
