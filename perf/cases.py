"""Timed cases: the work that a training program has this library do, through its public calls.

A case is a layer (or the seven layers of a decoder block), a representation (codebooks, codewords, group size, data
types), a subspace size and what is done with it:

  step    select -> re-encode -> dequantise: the V step and the dequantisation that opens the next step
  block   the same over every layer of a decoder block in one call
  trust   the V step whose subspace size follows from the trust ratio
  ste     Adam direction -> selection with a straight-through buffer -> re-encode against the buffer -> dequantise
  refine  a step of an additive representation with the local search after the beam search
  pstep   the P step's half: gradients of codebooks and scales, Adam on both, dequantisation

Weights, updates, scales and codebooks follow the recipe of ``paper_2405_14852_b200.synth`` (W ~ N(0, 0.02^2),
g ~ N(0, 0.001^2), one scale per row, codewords sampled from the scaled groups), drawn on the GPU.
"""
from __future__ import annotations

import math

import torch

from paper_2405_14852_b200 import binding as B
from paper_2405_14852_b200.vstep import VStepLayer

LARGEST_PAIRS = 28672 * 1024 * 65536  # codeword pairs of the largest listed case
LARGEST_AREA = 28672 * 8192


def _case(op, rows, cols, *, M=1, K=65536, gd=8, cb="f16", out="f32", k=0, beam=8, name=None):
    c = {"op": op, "rows": rows, "cols": cols, "M": M, "K": K, "gd": gd, "cb": cb, "out": out, "k": k, "beam": beam}
    if name:
        c["name"] = name
    return c


def listed():
    block = _case("block", 5120, 5120, out="f16", name="block13b_1x16")  # rows = cols = hidden size
    block.update(kv=5120, ffn=13824, k=100)  # k: one group in so many
    return [
        # the smallest layer of the benchmark table, every group: a call whose launches are all it costs
        _case("step", 256, 256, K=256, cb="f32", k=8192, name="tiny_1x8_f32"),
        # the usual training step on one attention projection: one 16-bit codebook, one group in a hundred
        _case("step", 4096, 4096, k=20971, name="attn7b_1x16"),
        # the same with two 8-bit codebooks and beam search, on a feed-forward projection
        _case("step", 11008, 4096, M=2, K=256, k=56360, name="mlp7b_2x8"),
        # one decoder block per call, W_hat in half precision for the forward pass
        block,
        # the largest: every group of the largest projection is re-encoded (as after initialisation)
        _case("step", 28672, 8192, k=28672 * 1024, name="gate70b_1x16_full"),
        # nothing a multiple of anything: odd rows and groups per row, a codebook that is not full, a narrow beam
        _case("refine", 3001, 4104, M=2, K=251, k=20011, beam=5, name="ragged_2x8_refine"),
        # three additive codebooks
        _case("step", 11008, 4096, M=3, K=256, out="f16", k=56360, name="mlp7b_3x8"),
        # groups of 16 weights
        _case("step", 4096, 4096, gd=16, out="f16", k=10485, name="attn7b_g16_1x16"),
        # subspace size from the trust ratio, capped at one group in a hundred
        _case("trust", 4096, 4096, k=20971, name="attn7b_1x16_trust"),
        # P step with a large codebook, and with two small ones
        _case("pstep", 4096, 4096, name="attn7b_1x16_pstep"),
        _case("pstep", 11008, 4096, M=2, K=256, out="f16", name="mlp7b_2x8_pstep"),
        # the update direction of the paper's training runs with the straight-through buffer
        _case("ste", 5120, 5120, M=2, K=256, out="f16", k=32768, name="attn13b_2x8_ste"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(("step", "step", "step", "step", "block", "trust", "ste", "refine", "pstep"))
    gd = 16 if op != "refine" and rng.random() < 0.12 else 8
    M = 1 if gd == 16 else rng.choice((2, 2, 3, 4)) if op == "refine" else rng.choice((1, 1, 1, 2, 2, 3, 4))
    cb = "f32" if gd == 8 and rng.random() < 0.15 else "f16"
    K = rng.randint(64, 256) if M > 1 else _log_int(rng, 4096 if gd == 16 else 256, 65536 if cb == "f16" else 4096)
    if M > 1 and rng.random() < 0.5:
        K = 256
    rows, per_row = _log_int(rng, 256, 28672), _log_int(rng, 32, 28672 // gd)
    most = {"step": LARGEST_AREA, "block": 5120, "trust": 2 ** 25, "ste": 2 ** 25, "refine": 2 ** 26, "pstep": 2 ** 26}[op]
    if op == "block":
        per_row = _log_int(rng, 64, most // gd)
        rows = per_row * gd
    while rows * per_row * gd > most and op != "block":
        if rows > per_row * gd:
            rows = max(256, rows // 2 + rng.randint(0, 1))
        else:
            per_row = max(32, per_row // 2 + rng.randint(0, 1))
    G = rows * per_row
    K = min(K, G // M)
    c = _case(op, rows, per_row * gd, M=M, K=K, gd=gd, cb=cb, out=rng.choice(("f16", "f32")),
              beam=rng.choice((8, 8, 8, rng.randint(1, 7))))
    if op == "block":
        c["kv"] = max(1, per_row // rng.choice((1, 2, 4, 8))) * gd
        c["ffn"] = int(per_row * rng.uniform(2.5, 4.0)) * gd
        c["K"] = min(c["K"], c["kv"] * per_row // M)
        c["k"] = rng.choice((1000, 100, 100, 30))
    elif op != "pstep":
        tau = math.exp(rng.uniform(math.log(0.001), math.log({"step": 1.0, "refine": 0.1, "trust": 0.05, "ste": 0.1}[op])))
        # the slower formats are taken with fewer groups, so that no drawn case costs more than the largest listed one
        weight = 2 if M == 1 and cb == "f16" and K >= 1024 else 8 if M == 1 else 16 if M == 2 else 40
        c["k"] = max(1, min(int(tau * G), LARGEST_PAIRS // (weight * _pairs(c))))
    return c


# ---- inputs ------------------------------------------------------------------------------------------------------------


def _shapes(c):
    if c["op"] != "block":
        return [(c["rows"], c["cols"])]
    h, kv, f = c["rows"], c["kv"], c["ffn"]
    return [(h, h), (kv, h), (kv, h), (h, h), (f, h), (f, h), (h, f)]


def _codebooks(c, W, scale, gen):
    """[M, K, gd]: codewords sampled from the scaled groups, each further codebook from what the earlier ones leave."""
    gd, K = c["gd"], c["K"]
    per_row = W.shape[1] // gd
    pick = torch.randperm(W.shape[0] * per_row, generator=gen, device="cuda")
    groups, books = W.view(-1, gd), []
    for m in range(c["M"]):
        ids = pick[m * K:(m + 1) * K]
        X = groups[ids] / scale[ids // per_row, None]
        for book in books:
            X = X - book[torch.cdist(X, book).argmin(1)]
        X = X if m == 0 else 0.3 * X
        books.append(X.half().float() if c["cb"] == "f16" else X)
    return torch.stack(books).to(torch.float16 if c["cb"] == "f16" else torch.float32).contiguous()


def _layer(c, rows, cols, k, eta, gen):
    W = torch.randn(rows, cols, generator=gen, device="cuda").mul_(0.02)
    g = torch.randn(rows, cols, generator=gen, device="cuda").mul_(1e-3)
    scale = W.abs().amax(1)
    books = _codebooks(c, W, scale, gen)
    codes = torch.randint(0, c["K"], (W.numel() // c["gd"], c["M"]), generator=gen, device="cuda")
    codes = codes.to(torch.uint8 if c["K"] <= 256 else torch.int16)
    return VStepLayer(rows, cols, W, g, scale, books, codes, eta=eta, beam=c["beam"], max_k=k, group_dim=c["gd"])


def _encode_all(layer):
    """Codes as an earlier V step over every group leaves them."""
    every = VStepLayer(layer.rows, layer.cols, layer.W, layer.g, layer.scale, layer.codebooks, layer.codes, eta=0.0,
                       beam=layer.beam, group_dim=layer.group_dim)
    every.encode(torch.arange(layer.num_groups, dtype=torch.int32, device="cuda"))


def prepare(c, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dtype = torch.float16 if c["out"] == "f16" else torch.float32
    s = {"op": c["op"], "k": c["k"]}
    if c["op"] == "block":
        layers, ks = [], []
        for rows, cols in _shapes(c):
            ks.append(max(1, rows * cols // c["gd"] // c["k"]))
            layers.append(_layer(c, rows, cols, None, 1.0, gen))
        s["layers"] = layers
        s["idx"] = [torch.empty(k, dtype=torch.int32, device="cuda") for k in ks]
        s["W_hat"] = [torch.empty(x.rows, x.cols, dtype=dtype, device="cuda") for x in layers]
        s["block"] = B.Block([x.desc for x in layers], ks, s["idx"], s["W_hat"])
        s["ws"] = torch.empty(s["block"].workspace_bytes(), dtype=torch.uint8, device="cuda")
        B.pvt_workspace_init(s["ws"])
        return s
    eta = 1e-5 if c["op"] == "ste" else 1.0  # ste: the codes' learning rate, on an Adam-normalised direction
    L = s["layer"] = _layer(c, c["rows"], c["cols"], c["k"] or None, eta, gen)
    s["W_hat"] = torch.empty(L.rows, L.cols, dtype=dtype, device="cuda")
    if c["op"] != "pstep" and c["op"] != "trust":
        s["idx"] = torch.empty(c["k"], dtype=torch.int32, device="cuda")
    if c["op"] in ("trust", "pstep"):
        _encode_all(L)
    if c["op"] == "refine":
        s["err"] = torch.empty(c["k"], dtype=torch.float32, device="cuda")
        s["moves"] = torch.empty(c["k"], dtype=torch.int32, device="cuda")
    if c["op"] == "ste":
        # the gradients of four batches, one after the other; moments as some steps of training leave them
        s["grads"] = [L.g] + [torch.randn(L.rows, L.cols, generator=gen, device="cuda").mul_(1e-3) for _ in range(3)]
        s["avg"] = sum(s["grads"]) * 0.25
        s["avg_sq"] = sum(x * x for x in s["grads"]) * 0.25
        s["buffer"] = L.W.clone()
        s["dir"] = torch.empty_like(L.W)
        s["by_dir"] = VStepLayer(L.rows, L.cols, L.W, s["dir"], L.scale, L.codebooks, L.codes, eta=eta, beam=c["beam"],
                                 max_k=c["k"], group_dim=c["gd"])
        s["turn"] = 0
    if c["op"] == "pstep":
        # master copies in single precision; a half-precision codebook is refreshed from its master copy
        s["books"] = L.codebooks.float() if c["cb"] == "f16" else L.codebooks
        s["grad_books"] = torch.empty(L.codebooks.shape, dtype=torch.float64, device="cuda")
        s["grad_scale"] = torch.empty(L.rows, dtype=torch.float64, device="cuda")
        s["books_m"], s["books_v"] = torch.zeros_like(s["books"]), torch.zeros_like(s["books"])
        s["scale_m"], s["scale_v"] = torch.zeros_like(L.scale), torch.zeros_like(L.scale)
        s["t"] = 0
    return s


# ---- one pass ----------------------------------------------------------------------------------------------------------


def run(s):
    op = s["op"]
    if op == "block":
        B.pvt_vstep_block(s["block"], s["ws"])
        return {"idx": s["idx"], "codes": [x.codes for x in s["layers"]], "W_hat": s["W_hat"]}
    L, k, W_hat = s["layer"], s["k"], s["W_hat"]
    if op == "step":
        L.step(k, s["idx"], W_hat)
        return {"idx": s["idx"], "codes": L.codes, "W_hat": W_hat}
    if op == "trust":
        idx, n, stats = L.step_trust(k, 0.01)
        L.dequant(W_hat)
        return {"idx": idx, "n": n, "stats": stats, "codes": L.codes, "W_hat": W_hat}
    if op == "refine":
        L.select(k, s["idx"])
        L.encode(s["idx"], s["err"])
        B.pvt_vstep_refine(L.desc, s["idx"], k, 16, s["err"], s["moves"])
        L.dequant(W_hat)
        return {"idx": s["idx"], "codes": L.codes, "err": s["err"], "moves": s["moves"], "W_hat": W_hat}
    if op == "ste":
        grad = s["grads"][s["turn"] % 4]
        s["turn"] += 1
        B.pvt_adam_direction(grad, s["avg"], s["avg_sq"], s["dir"], 100 + s["turn"])
        V = s["by_dir"]
        V.select_ste(s["buffer"], k, s["idx"])
        V.encode_against(s["buffer"], s["idx"])
        V.dequant(W_hat)
        return {"idx": s["idx"], "codes": L.codes, "W_hat": W_hat, "buffer": s["buffer"], "dir": s["dir"],
                "avg": s["avg"], "avg_sq": s["avg_sq"]}
    s["t"] += 1
    B.pvt_pstep_grad(L.desc, s["grad_books"], s["grad_scale"])
    half = L.codebooks if L.codebooks.dtype == torch.float16 else None
    B.pvt_adam_update(s["books"], s["grad_books"], s["books_m"], s["books_v"], s["t"], 1e-6, param_f16=half)
    B.pvt_adam_update(L.scale, s["grad_scale"], s["scale_m"], s["scale_v"], s["t"], 1e-6)
    L.dequant(W_hat)
    return {"grad_books": s["grad_books"], "grad_scale": s["grad_scale"], "books": s["books"], "scale": L.scale,
            "codebooks": L.codebooks, "books_m": s["books_m"], "books_v": s["books_v"], "scale_m": s["scale_m"],
            "scale_v": s["scale_v"], "W_hat": W_hat}


# ---- what a pass cannot do without -------------------------------------------------------------------------------------


def _pairs(c):
    """Codeword evaluations per re-encoded group, as the definition of the search counts them."""
    return c["K"] if c["M"] == 1 else c["K"] + c["beam"] * c["K"] * (c["M"] - 1)


def work(c):
    gd, M, K = c["gd"], c["M"], c["K"]
    code, cw, out = M * (1 if K <= 256 else 2), 2 if c["cb"] == "f16" else 4, 2 if c["out"] == "f16" else 4
    total, flops = 0, 0
    for rows, cols in _shapes(c):
        n, G = rows * cols, rows * cols // gd
        total += M * K * gd * cw + 4 * rows + G * code + out * n  # codebooks, scales, codes, W_hat
        if c["op"] == "pstep":
            # update; binary64 gradients out; parameters and moments in and out (and the half-precision codebook)
            total += 4 * n + (8 + 24) * (M * K * gd + rows) + (2 * M * K * gd if cw == 2 else 0)
            flops += 2 * n * M + 2 * n
            continue
        k = max(1, G // c["k"]) if c["op"] == "block" else c["k"]
        # update (all of it unless every group is taken anyhow), weights, indices and codes of the chosen groups
        total += 4 * n + 4 * gd * k + 4 * k + code * k
        if M == 1:
            flops += 2 * gd * K * k
        else:  # <t, c> once per codeword of every codebook, then one addition per kept partial tuple and codeword
            flops += (2 * gd * K * M + 2 * c["beam"] * K * (M - 1)) * k
        if c["op"] == "refine":
            total += 8 * k
        if c["op"] == "ste":
            total += 4 * n * 7  # moments and buffer in and out, direction out
    return {"bytes": total, "flops": flops}


def tolerance(c):
    if c["op"] == "pstep":
        # binary64 sums in any order, rounded once to binary32 for Adam; a half-precision value may round the other way
        return {"rel": 1e-5, "max": 2e-3, "differ": 0.0}
    if c["op"] == "trust":
        return {"rel": 1e-9, "max": 1e-9, "differ": 0.0}  # two binary64 sums; everything else is the same to the bit
    return "exact"
