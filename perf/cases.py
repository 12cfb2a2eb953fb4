"""Workloads of the compressed linear layer, as programs that use the library run them.

Two kinds of case:

``forward``   one call of one layer, Y = X (s Q)^T + (X R^T) L^T, on weights packed once.  The program
              keeps the packed weight (and, where ``slim_decode_layout_hint`` asks for it, the
              decode-tiled copy), the adapters (bf16, or int4 codes with group scales) and a
              workspace; every call gets an activation batch and returns a new Y.
``compress``  one layer's compression: float32 weights -> SLiM-Quant codes and scale -> 2:4 mask ->
              packed weight, and its two adapters -> int4 codes.

Layer shapes are the LLaMA-2 7B / 13B / 70B linears, whole or as one rank's shard when the MLP's
inner dimension is split over 2, 4 or 8 GPUs (those are multiples of 64 or 128 and of nothing larger).
"""
from __future__ import annotations

import math

import torch

from paper_2410_09615_b200 import binding as K
from paper_2410_09615_b200.inputs import rank_for_ratio

_GROUP = 128                      # adapter elements that share one scale


def _forward(name, d_in, d_out, b, r, adapters="bf16"):
    return {"name": name, "op": "forward", "d_in": d_in, "d_out": d_out, "b": b, "r": r, "adapters": adapters}


def listed():
    return [
        # the smallest call the library is configured for: eight tokens through a 512 x 512 layer
        _forward("fwd_512x512_b8", 512, 512, 8, 64),
        # one user's decode step: attention projection of the 7B model
        _forward("fwd_4096x4096_b1", 4096, 4096, 1, 416),
        # one user's decode step: the largest layer of the 70B model (gate / up)
        _forward("fwd_8192x28672_b1", 8192, 28672, 1, 832),
        # decode step of sixteen users: the 70B model's down projection
        _forward("fwd_28672x8192_b16", 28672, 8192, 16, 832),
        # decode step of four users on one of two GPUs that share the 7B model's MLP (down, half of 11008)
        _forward("fwd_5504x4096_b4", 5504, 4096, 4, 416),
        # decode step of sixteen users: the 70B model's k / v projection with int4 adapters
        _forward("fwd_q_8192x1024_b16", 8192, 1024, 16, 112, "int4"),
        # decode step of a busy server, or a very short prompt: 64 tokens through the 13B gate / up layer
        _forward("fwd_5120x13824_b64", 5120, 13824, 64, 512),
        # a short prompt of no round length through a 70B attention projection without adapters
        _forward("fwd_8192x8192_b333_r0", 8192, 8192, 333, 0),
        # an ordinary prompt: 2048 tokens through the 7B gate / up layer
        _forward("fwd_4096x11008_b2048", 4096, 11008, 2048, 416),
        # the largest: 4096 tokens through the 70B down projection
        _forward("fwd_28672x8192_b4096", 28672, 8192, 4096, 832),
        # a prompt on one of eight GPUs that share the 13B model's MLP (down, an eighth of 13824), int4 adapters
        _forward("fwd_q_1728x5120_b600", 1728, 5120, 600, 176, "int4"),
        # compressing a layer: 7B gate / up
        {"name": "compress_4096x11008", "op": "compress", "d_in": 4096, "d_out": 11008, "r": 416},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, lo, hi, step):
    return min(hi, max(lo, int(round(_log_uniform(rng, lo, hi) / step)) * step))


# (d_in, d_out) of the layers, and of one rank's shard of an MLP layer
_WHOLE = [(4096, 4096), (4096, 11008), (11008, 4096), (5120, 5120), (5120, 13824), (13824, 5120),
          (8192, 8192), (8192, 1024), (8192, 28672), (28672, 8192)]
_SHARDS = [(5504, 4096), (4096, 5504), (2752, 4096), (4096, 2752), (6912, 5120), (5120, 6912), (3456, 5120), (5120, 3456),
           (1728, 5120), (5120, 1728), (3584, 8192), (8192, 3584)]


def draw(rng):
    if rng.random() < 0.12:
        d_in, d_out = rng.choice([(_size(rng, 1024, 8192, 64), _size(rng, 1024, 11008, 16)), rng.choice(_SHARDS)])
        return {"op": "compress", "d_in": d_in, "d_out": d_out, "r": rank_for_ratio(rng.choice([0.05, 0.1, 0.2]), d_in, d_out)}
    kind = rng.random()
    if kind < 0.4:
        d_in, d_out = rng.choice(_WHOLE)
    elif kind < 0.65:
        d_in, d_out = rng.choice(_SHARDS)
    else:                         # any width the packed format takes
        d_in, d_out = _size(rng, 512, 8192, 64), _size(rng, 512, 8192, 16)
    # half of the calls are decode steps, the others prompts and large batches
    b = rng.randint(1, 16) if rng.random() < 0.5 else int(_log_uniform(rng, 17, 4096))
    if kind >= 0.4:
        b = min(b, 1024)
    r = rank_for_ratio(rng.choice([0.0, 0.05, 0.1, 0.1, 0.1, 0.2]), d_in, d_out)
    return {"op": "forward", "d_in": d_in, "d_out": d_out, "b": b, "r": r,
            "adapters": "int4" if r and rng.random() < 0.3 else "bf16"}


def _normal(shape, std, gen, dtype):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).mul_(std).to(dtype)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    d_in, d_out, r = case["d_in"], case["d_out"], case["r"]
    W = _normal((d_out, d_in), 0.02, gen, torch.float32)
    xbar = torch.rand(d_in, generator=gen, device="cuda", dtype=torch.float32).add_(0.5)   # average input magnitudes
    L = _normal((d_out, r), 0.02, gen, torch.bfloat16) if r else None
    R = _normal((r, d_in), 0.02, gen, torch.bfloat16) if r else None
    if case["op"] == "compress":
        return {"op": "compress", "W": W, "xbar": xbar, "L": L, "R": R}
    b = case["b"]
    codes, scale, _, _ = K.slim_quant(W)
    vals, meta = K.slim_pack(codes, K.slim_mask_top2(codes, xbar))
    state = {"op": "forward", "X": _normal((b, d_in), 1.0, gen, torch.bfloat16), "s": float(scale[0]), "d_out": d_out,
             "vals": vals, "meta": meta, "L": L, "R": R}
    if case["adapters"] == "int4":
        state["op"] = "forward_q"
        state["Lq"], state["Ls"] = K.slim_pack_adapter(L)
        state["Rq"], state["Rs"] = K.slim_pack_adapter(R)
        del state["L"], state["R"]
        state["ws"] = torch.empty(K.slim_workspace_bytes_q(b, d_out, d_in, r), dtype=torch.uint8, device="cuda")
        K.slim_workspace_reset(state["ws"])
        return state
    state["ws"] = K.new_workspace(b, d_out, d_in, r)
    if K.slim_decode_layout_hint(b, d_out, d_in, r) == K.LAYOUT_DECODE_TILED:
        state["op"] = "forward_tiled"
        state["tiled"] = K.slim_repack_tiled(vals, meta)
        del state["vals"], state["meta"]
    return state


def run(st):
    op = st["op"]
    if op == "forward":
        return K.slim_linear_fwd(st["X"], st["vals"], st["meta"], st["s"], st["L"], st["R"], workspace=st["ws"])
    if op == "forward_tiled":
        return K.slim_linear_fwd_tiled(st["X"], st["tiled"], st["d_out"], st["s"], st["L"], st["R"], workspace=st["ws"])
    if op == "forward_q":
        return K.slim_linear_fwd_q(st["X"], st["vals"], st["meta"], st["s"], st["Lq"], st["Ls"], st["Rq"], st["Rs"],
                                   workspace=st["ws"])
    codes, scale_alpha, table, _ = K.slim_quant(st["W"])
    vals, meta = K.slim_pack(codes, K.slim_mask_top2(codes, st["xbar"]))
    Lq, Ls = K.slim_pack_adapter(st["L"])
    Rq, Rs = K.slim_pack_adapter(st["R"])
    return {"codes": codes, "scale_alpha": scale_alpha, "table": table, "vals": vals, "meta": meta,
            "Lq": Lq, "Ls": Ls, "Rq": Rq, "Rs": Rs}


def _adapter_bytes(rows, cols, kind):
    return 2 * rows * cols if kind == "bf16" else rows * (cols // 2 + 2 * math.ceil(cols / _GROUP))


def work(case):
    d_in, d_out, r = case["d_in"], case["d_out"], case["r"]
    packed = 0.375 * d_out * d_in
    if case["op"] == "compress":
        read = 4 * d_out * d_in + 4 * d_in + _adapter_bytes(d_out, r, "bf16") + _adapter_bytes(r, d_in, "bf16")
        written = d_out * d_in + packed + _adapter_bytes(d_out, r, "int4") + _adapter_bytes(r, d_in, "int4")
        return {"bytes": read + written, "flops": 0}
    b = case["b"]
    adapters = _adapter_bytes(d_out, r, case["adapters"]) + _adapter_bytes(r, d_in, case["adapters"]) if r else 0
    # two kept weights of every four: d_in / 2 multiply-adds per output, and the two thin adapter products
    return {"bytes": packed + adapters + 2 * b * (d_in + d_out), "flops": b * d_in * d_out + 2 * b * r * (d_in + d_out)}


def tolerance(case):
    if case["op"] == "compress":
        return "exact"            # codes, bytes and the scale search's decisions are defined bit for bit
    # bf16 output, and the rank-r intermediate rounded to bf16 once
    return {"rel": 1e-2, "max": 3e-2}
