"""Timed workloads of the stage-boundary codec, through the torch-facing public API.

Every case is one thing a training program of the paper does at a pipeline stage, at a size from
this repository's workloads (synth.py), benchmark sweeps or the paper's own figures:

  step       one microbatch of a body stage: expand what arrives (decompress), compress what leaves,
             and the same two steps for the activation gradients of the backward pass
  compress, decompress, backward   the directions of that step by themselves
  wire       the same step with the rows that really cross the link: fp32 words with the token id,
             and the last residual add fused into compress
  reproject  the original SSN: every constrained weight of a stage after an optimizer step
  reparam    a reparameterised projection layer: output, activation gradient, factor gradient
  average    an averaging round of a stage's parameters and the stage-wise clipping of its gradients

The cases differ in what bounds them: a few thousand tokens (launches and latency), a microbatch that
barely fills the GPU, one that streams for a hundred microseconds; bf16 and fp32 storage; whole sequences
with implicit positions, packed documents with explicit ones, models without a positional table; ranks
that are no multiple of 8, stored packed or padded.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_13332_b200 import dp_ops, synth
from paper_2607_13332_b200.runner import Codec, padded_columns

_TORCH = {"bf16": torch.bfloat16, "f32": torch.float32}
_BYTES = {"bf16": 2, "f32": 4}
_TOKEN_KINDS = ("step", "compress", "decompress", "backward", "wire")


def _tokens(kind, d, k, tokens, seq, vocab, ids="zipf", dtype="bf16", positions="implicit", tables=False, padded=False):
    """A case over tokens.  positions: "implicit" (tokens = whole sequences of length seq), "packed"
    (documents of unequal length, at most seq, with an explicit position per token) or "none"."""
    return {"kind": kind, "d": d, "k": k, "tokens": tokens, "seq": seq, "vocab": vocab, "ids": ids, "dtype": dtype,
            "positions": positions, "tables": tables, "padded": padded}


def listed():
    tiny, mid, big = synth.TINY, synth.MID, synth.STAGE_8B
    cases = {
        # the smallest workload: four fp32 calls of a few microseconds each, launches and host time count
        "tiny_fp32_step": _tokens("step", tiny.d, tiny.k, tiny.n_tokens, tiny.seq_len, tiny.vocab, tiny.ids_law, "f32"),
        # one sequence per call, the smallest microbatch of the wide model
        "one_sequence_step": _tokens("step", big.d, big.k, big.seq_len, big.seq_len, big.vocab),
        # the mid-size model's microbatch
        "mid_step": _tokens("step", mid.d, mid.k, mid.n_tokens, mid.seq_len, mid.vocab, mid.ids_law),
        # packed documents: an odd number of tokens, explicit positions, rank 40 of 2048
        "packed_documents_step": _tokens("step", 2048, 40, 10007, 2048, mid.vocab, positions="packed"),
        # a boundary kept in fp32
        "fp32_step": _tokens("step", 2048, 40, 8192, 1024, mid.vocab, dtype="f32"),
        # the wide model's large microbatch, sender and receiver of the forward pass and the backward pass
        "stage_compress": _tokens("compress", big.d, big.k, big.n_tokens, big.seq_len, big.vocab),
        "stage_decompress": _tokens("decompress", big.d, big.k, big.n_tokens, big.seq_len, big.vocab),
        "stage_backward": _tokens("backward", big.d, big.k, big.n_tokens, big.seq_len, big.vocab),
        # three coalesced sequences of 4096 tokens as fp32 wire rows, rank 51 of 5120, no positional
        # table (rotary positions), the basis stored as it is
        "wire_rank51": _tokens("wire", 5120, 51, 3 * 4096, 4096, big.vocab, positions="none"),
        # the output projections of two blocks after an optimizer step
        "reproject_two_blocks": {"kind": "reproject", "d": 4096, "k": 40, "layers": 2, "down": 14336, "side": "right",
                                 "dtype": "bf16", "padded": False},
        # the reparameterised down-projection, forward and backward
        "reparam_down_proj": {"kind": "reparam", "d": 4096, "k": 40, "m": 14336, "tokens": 16384, "dtype": "bf16",
                              "padded": False},
        # one round over the 5 % segment of four blocks' parameters, three senders, and their clipping
        "averaging_round": {"kind": "average", "d": 4096, "layers": 4, "senders": 3, "round": 7, "grads": "bf16", "clips": True},
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        case = _draw_any(rng)
        if _cost(case) <= most:
            return case


def _cost(case):
    """Comparable cost of a pass: its bytes, or its operations where those weigh more (fp32 ones do)."""
    w = work(case)
    return max(w["bytes"], w["flops"] / (3 if case.get("dtype") == "f32" else 20))


def _draw_any(rng):
    kind = rng.choice(_TOKEN_KINDS * 2 + ("step",) * 4 + ("reproject", "reparam", "average"))
    if kind == "average":
        return {"kind": kind, "d": rng.choice((512, 1024, 2048, 4096)), "layers": rng.randint(1, 4), "senders": rng.randint(1, 6),
                "round": rng.randint(0, 60), "grads": rng.choice(("bf16", "f32")), "clips": rng.random() < 0.5}
    d = rng.choice((512, 768, 1024, 1536, 2048, 2048, 2560, 3072, 4096, 4096, 5120, 8192))
    # ranks of the sweeps, or anything up to 128
    k = rng.choice((8, 16, 32, 40, 64, 128)) if rng.random() < 0.5 else _log(rng, 8, 128)
    dtype = "f32" if rng.random() < 0.2 else "bf16"
    padded = rng.random() < 0.5
    if kind == "reproject":
        return {"kind": kind, "d": d, "k": k, "layers": rng.randint(1, 4), "down": d * 7 // 2, "side": rng.choice(("left", "right")),
                "dtype": dtype, "padded": padded}
    if kind == "reparam":
        return {"kind": kind, "d": d, "k": k, "m": rng.choice((d, d * 7 // 2, 4 * d)), "tokens": _log(rng, 512, 32768), "dtype": dtype,
                "padded": padded}
    vocab = rng.choice((1024, 32000, 128256))
    ids = rng.choice(("zipf", "uniform"))
    positions = rng.choice(("implicit", "implicit", "packed", "none"))
    seq = rng.choice((512, 1024, 2048, 4096)) if rng.random() < 0.7 else rng.randint(300, 4096)
    tokens = _log(rng, 512, 65536)
    if positions == "implicit":
        tokens = max(1, round(tokens / seq)) * seq
    return _tokens(kind, d, k, tokens, seq, vocab, ids, dtype, positions, kind in ("step", "compress", "wire") and rng.random() < 0.25, padded)


# ---- inputs ------------------------------------------------------------------------------------
def _normal(g, shape, std, dtype):
    return torch.empty(shape, device="cuda", dtype=dtype).normal_(0.0, std, generator=g)


def _basis(g, d, k, dtype, padded):
    q = torch.linalg.qr(_normal(g, (d, k), 1.0, torch.float32))[0].to(dtype).contiguous()
    return padded_columns(q) if padded else q


def _ids(g, case):
    v, n = case["vocab"], case["tokens"]
    if case["ids"] == "uniform":
        return torch.randint(0, v, (n,), device="cuda", dtype=torch.int32, generator=g)
    p = torch.arange(1, v + 1, device="cuda", dtype=torch.float64).pow_(-1.1)
    rank = torch.multinomial(p, n, replacement=True, generator=g)
    return torch.randperm(v, device="cuda", generator=g)[rank].to(torch.int32)


def _packed_positions(g, case):
    """Positions of documents laid end to end, lengths from 16 to seq."""
    n, seq = case["tokens"], case["seq"]
    u = torch.rand(n // 16 + 1, device="cuda", generator=g)
    lengths = torch.exp(math.log(16) + u * math.log(seq / 16)).long().clamp_(16, seq)
    ends = lengths.cumsum(0)
    t = torch.arange(n, device="cuda")
    doc = torch.searchsorted(ends, t, right=True)
    return (t - (ends - lengths)[doc]).to(torch.int32)


def _sinusoid(seq, d, dtype):
    p = torch.arange(seq, device="cuda", dtype=torch.float32)[:, None]
    i = torch.arange(d, device="cuda", dtype=torch.float32)[None, :]
    angle = p * torch.exp(-math.log(10000.0) * 2.0 * torch.floor(i / 2) / d)
    return torch.where(i % 2 == 0, torch.sin(angle), torch.cos(angle)).to(dtype)


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return {"kind": case["kind"], **(_prepare_tokens if case["kind"] in _TOKEN_KINDS else _PREPARE[case["kind"]])(case, g)}


def _prepare_tokens(case, g):
    kind, d, k, n, seq, dt = (case[x] for x in ("kind", "d", "k", "tokens", "seq", "dtype"))
    tdt = _TORCH[dt]
    U = _basis(g, d, k, tdt, case["padded"])
    s = {"ids": _ids(g, case), "seq": seq, "pos": None, "codec": None, "plain": Codec(dt, U)}
    P = None
    if case["positions"] != "none":
        P = _sinusoid(seq, d, tdt)
    if case["positions"] == "packed":
        s["pos"] = _packed_positions(g, case)
    E = _normal(g, (case["vocab"], d), 0.02, tdt)
    s["codec"] = Codec(dt, U, E, P)
    if case["tables"]:
        s["codec"].prepare_tables()
    if kind in ("step", "compress", "wire"):   # a hidden state: shift rows, a point of the subspace, a little noise
        X = _normal(g, (n, k), 1.0, torch.float32) @ U.float().T
        X += E[s["ids"]]
        if P is not None:
            X += P[s["pos"].long() if s["pos"] is not None else torch.arange(n, device="cuda") % seq]
        X += _normal(g, (n, d), 0.05, tdt)
        s["X"] = X.to(tdt)
    if kind == "wire":                         # the residual stream before the last block, and that block's output
        s["R"] = _normal(g, (n, d), 0.3, tdt)
        wire = torch.empty((n, k + 1), dtype=torch.int32, device="cuda")
        wire[:, :k] = _normal(g, (n, k), 1.0, torch.float32).view(torch.int32)
        wire[:, k] = s["ids"]
        s["wire"] = wire
        s["wire_grad"] = _normal(g, (n, k), 1e-2, torch.float32).view(torch.int32)
    if kind in ("step", "decompress"):
        s["Z"] = _normal(g, (n, k), 1.0, tdt)
    if kind in ("step", "backward"):
        s["dZ"] = _normal(g, (n, k), 1e-2, tdt)
    if kind in ("step", "backward", "wire"):
        s["G"] = _normal(g, (n, d), 1e-2, tdt)
    if case["padded"] and "Z" in s:
        s["Z"] = padded_columns(s["Z"])
    if case["padded"] and "dZ" in s:
        s["dZ"] = padded_columns(s["dZ"])
    return s


def _prepare_reproject(case, g):
    d, tdt = case["d"], _TORCH[case["dtype"]]
    rows = [d, case["down"]] * case["layers"]
    return {"codec": Codec(case["dtype"], _basis(g, d, case["k"], tdt, case["padded"])), "side": case["side"],
            "weights": [_normal(g, (r, d) if case["side"] == "right" else (d, r), 0.02, tdt) for r in rows]}


def _prepare_reparam(case, g):
    d, k, m, n, tdt = case["d"], case["k"], case["m"], case["tokens"], _TORCH[case["dtype"]]
    U = _basis(g, d, k, tdt, case["padded"])
    Zw = _normal(g, (m, k), 0.02, tdt)
    Zw = padded_columns(Zw) if case["padded"] else Zw
    return {"codec": Codec(case["dtype"], U), "transposed": Codec(case["dtype"], Zw), "U": U, "Zw": Zw,
            "H": _normal(g, (n, m), 1.0, tdt), "dY": _normal(g, (n, d), 1e-2, tdt)}


def _stage_shapes(case):
    """Parameter tensors of a stage: attention and MLP projections and norms of every block."""
    d, f = case["d"], case["d"] * 7 // 2
    return [(d, d)] * 4 * case["layers"] + [(f, d)] * 3 * case["layers"] + [(d,)] * 2 * case["layers"]


def _prepare_average(case, g):
    shapes = _stage_shapes(case)
    n = sum(math.prod(s) for s in shapes)
    lo, hi = dp_ops.sparta_segment(n, 20, case["round"])
    # gradient norm about 10 (clipped) or 0.1 (inside the budget)
    std = (10.0 if case["clips"] else 0.1) / math.sqrt(n)
    buf = _normal(g, (n,), 0.02, torch.float32)
    return {"buf": buf, "theta": buf + 1e-4, "acc": torch.zeros(hi - lo, device="cuda"), "n": n, "round": case["round"],
            "chunks": [_normal(g, (hi - lo,), 0.02, torch.float32) for _ in range(case["senders"])],
            "weights": [float(1 + i) for i in range(case["senders"])],
            "grads": [_normal(g, s, std, _TORCH[case["grads"]]) for s in shapes]}


_PREPARE = {"reproject": _prepare_reproject, "reparam": _prepare_reparam, "average": _prepare_average}


# ---- passes ------------------------------------------------------------------------------------
def run(s):
    return _RUN[s["kind"]](s)


def _run_compress(s):
    return s["codec"].compress(s["X"], s["ids"], seq_len=s["seq"], pos=s["pos"])


def _run_decompress(s):
    return s["codec"].decompress(s["Z"], s["ids"], seq_len=s["seq"], pos=s["pos"])


def _run_backward(s):
    return s["plain"].decompress(s["dZ"]), s["plain"].grad_project(s["G"])


def _run_step(s):
    return (_run_decompress(s), _run_compress(s), *_run_backward(s))


def _run_wire(s):
    codec, k = s["codec"], s["codec"].k
    X = codec.decompress_wire(s["wire"], seq_len=s["seq"], pos=s["pos"], with_ids=True)
    out = codec.compress_sum(s["X"], s["R"], s["ids"], seq_len=s["seq"], pos=s["pos"], wire=True, with_ids=True)
    dX = s["plain"].decompress_wire(s["wire_grad"])
    dZ = s["plain"].grad_project_wire(s["G"])
    return X, out.view(torch.float32)[:, :k], out[:, k], dX, dZ


def _run_reproject(s):
    s["codec"].weight_reproject_list(s["weights"], s["side"])
    return s["weights"]


def _run_reparam(s):
    Y = s["codec"].reparam_project(s["H"], s["Zw"])
    dH = s["transposed"].reparam_project(s["dY"], s["U"])
    return Y, dH, s["codec"].reparam_grad_factor(s["H"], s["dY"])


def _run_average(s):
    buf, theta, acc = s["buf"], s["theta"], s["acc"]
    lo, hi = dp_ops.sparta_segment(s["n"], 20, s["round"])
    snap = dp_ops.sparta_snapshot(buf, lo, hi)
    acc.zero_()
    for chunk, w in zip(s["chunks"], s["weights"]):
        dp_ops.sparta_accumulate(acc, chunk, w)
    deltas = dp_ops.sparta_deltas(acc, sum(s["weights"]), s["chunks"])
    dp_ops.sparta_add_delta(buf, lo, hi, deltas[0])
    dp_ops.sparta_apply_round(theta, lo, hi, buf[lo:hi], snap)
    norm2 = dp_ops.stage_clip(s["grads"], 0.3779)
    return snap, acc, deltas, buf, theta, norm2, s["grads"]


_RUN = {"compress": _run_compress, "decompress": _run_decompress, "backward": _run_backward, "step": _run_step, "wire": _run_wire,
        "reproject": _run_reproject, "reparam": _run_reparam, "average": _run_average}


# ---- the same passes in 64 bits, as plain torch ------------------------------------------------
def exact(case, seed):
    s = prepare(case, seed)
    return (_exact_tokens if case["kind"] in _TOKEN_KINDS else _EXACT[case["kind"]])(case, s)


def _exact_tokens(case, s):
    kind, n, k = case["kind"], case["tokens"], case["k"]
    codec = s["codec"]
    U = codec.U.double()

    def shift(rows):
        t = codec.E[s["ids"][rows]].double()
        if codec.P is not None:
            pos = s["pos"][rows] if s["pos"] is not None else torch.arange(rows.start, rows.stop, device="cuda") % s["seq"]
            t += codec.P[pos.long()].double()
        return t

    def by_rows(f, cols):
        out = torch.empty((n, cols), device="cuda", dtype=torch.float64)
        for lo in range(0, n, 8192):
            rows = slice(lo, min(n, lo + 8192))
            out[rows] = f(rows)
        return out

    def compress():
        return by_rows(lambda r: (s["X"][r].double() + (s["R"][r].double() if kind == "wire" else 0.0) - shift(r)) @ U, k)

    def expand(Z):
        return by_rows(lambda r: Z[r].double() @ U.T + shift(r), case["d"])

    def backward(dZ):
        return by_rows(lambda r: dZ[r].double() @ U.T, case["d"]), by_rows(lambda r: s["G"][r].double() @ U, k)

    if kind == "wire":
        X, out = expand(s["wire"][:, :k].view(torch.float32)), compress()
        return X, out, s["ids"], *backward(s["wire_grad"].view(torch.float32))
    if kind == "compress":
        return compress()
    if kind == "decompress":
        return expand(s["Z"])
    return backward(s["dZ"]) if kind == "backward" else (expand(s["Z"]), compress(), *backward(s["dZ"]))


def _exact_reproject(case, s):
    U = s["codec"].U.double()
    return [(w.double() @ U) @ U.T if case["side"] == "right" else U @ (U.T @ w.double()) for w in s["weights"]]


def _exact_reparam(case, s):
    U, Zw, dY = s["U"].double(), s["Zw"].double(), s["dY"].double()
    C, F = torch.empty((case["tokens"], case["k"]), device="cuda", dtype=torch.float64), 0.0
    dC = dY @ U
    for lo in range(0, case["tokens"], 4096):
        H = s["H"][lo:lo + 4096].double()
        C[lo:lo + 4096] = H @ Zw
        F = F + H.T @ dC[lo:lo + 4096]
    return C @ U.T, dC @ Zw.T, F


def _exact_average(case, s):
    n, r = s["n"], s["round"] % 20
    lo, hi = n * r // 20 & ~63, n if r == 19 else n * (r + 1) // 20 & ~63
    buf, theta = s["buf"].double(), s["theta"].double()
    snap = buf[lo:hi].clone()
    chunks = [c.double() for c in s["chunks"]]
    acc = sum(w * c for w, c in zip(s["weights"], chunks)) / sum(s["weights"])
    deltas = [acc - c for c in chunks]
    buf[lo:hi] += deltas[0]
    theta[lo:hi] += buf[lo:hi] - snap
    norm2 = sum(g.double().square().sum() for g in s["grads"])
    coef = min(1.0, 0.3779 / (math.sqrt(float(norm2)) + 1e-6))
    return snap, acc, deltas, buf, theta, norm2.reshape(1), [g.double() * coef for g in s["grads"]]


_EXACT = {"reproject": _exact_reproject, "reparam": _exact_reparam, "average": _exact_average}


# ---- what a pass cannot do without ------------------------------------------------------------
def _distinct_rows(case):
    """Expected number of distinct embedding rows among the tokens."""
    v, n = case["vocab"], case["tokens"]
    p = np.full(v, 1.0 / v) if case["ids"] == "uniform" else np.arange(1, v + 1, dtype=np.float64) ** -1.1
    return float(np.sum(-np.expm1(n * np.log1p(-p / p.sum()))))


def work(case):
    kind = case["kind"]
    if kind == "average":
        n = sum(math.prod(s) for s in _stage_shapes(case))
        seg, b = 4 * (n // 20), _BYTES[case["grads"]]
        # segment of buf in and out, snapshot out, chunks in, deltas and mean out, theta in and out
        return {"bytes": (6 + 2 * case["senders"]) * seg + n * b * (2 if case["clips"] else 1), "flops": 2 * n}
    d, k, b = case["d"], case["k"], _BYTES[case["dtype"]]
    if kind == "reproject":
        extent = case["layers"] * (d + case["down"])
        return {"bytes": 2 * extent * d * b + d * k * b, "flops": 4 * extent * d * k}
    n = case["tokens"]
    if kind == "reparam":
        # H and dY read by all three products once, Y and dH written; the factor gradient is fp32
        m = case["m"]
        return {"bytes": 2 * n * (m + d) * b + 2 * (m + d) * k * b + 4 * m * k, "flops": 2 * n * k * (3 * m + 3 * d)}
    shift = _distinct_rows(case) * d * b + 4 * n + (min(n, case["seq"]) * d * b if case["positions"] != "none" else 0)
    z = 4 if kind == "wire" else b
    one = n * d * b + n * k * z + d * k * b
    tables = (_distinct_rows(case) + min(n, case["seq"])) * k * 4 + 4 * n
    comp = one + (tables if case["tables"] else shift)
    w = {"compress": comp, "decompress": one + shift, "backward": 2 * one, "step": 3 * one + comp + shift,
         "wire": 3 * one + comp + shift + n * d * b}[kind]
    return {"bytes": w, "flops": 2 * n * d * k * {"compress": 1, "decompress": 1, "backward": 2}.get(kind, 4)}


def tolerance(case):
    """About four times what a comparison with fp64 sums shows: bf16 results differ by their output rounding
    (2^-9 on average, 3.9e-3 at most; the factor gradient also by the rounding of its bf16 coordinates, 8.2e-3),
    fp32 ones by sums of d products (2e-7, 1.7e-6 at most), of up to 32768 tokens for the factor gradient."""
    kind = case["kind"]
    if (case["grads"] if kind == "average" else case["dtype"]) == "bf16":
        return {"rel": 7e-3, "max": 3.2e-2 if kind == "reparam" else 1.6e-2}
    return {"rel": 1e-5, "max": 1e-4} if kind == "reparam" else {"rel": 2e-6, "max": 1.5e-5}
