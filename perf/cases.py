"""Timed cases of the library: what a user of Attention Pruning has it do, through the Python binding.

The procedure has three steps on the GPU (average the attention maps, select what is kept, run attention
under the kept entries) and retraining adds the derivative of the third.  A case is one call of a step
(one forward and one backward call for "train") on one shape:

  accumulate  ap_accumulate_attention   one calibration batch into the running sum
  mask        ap_build_mask[_layer]     selection -> element mask, tile list, counts
  fwd         ap_sparse_attention_fwd   inference under a pruned mask
  dense       ap_sparse_attention_fwd   inference under the unpruned list (ap_dense_tiles)
  train       ap_sparse_attention_fwd, ap_sparse_attention_bwd: one retraining pass of the attention
  entmax      ap_sparse_attention_entmax15_fwd  inference of a model normalised by 1.5-entmax

Shapes are those of the paper's experiments as inputs.py states them (encoder classification, language
modelling with and without memory keys, translation, 4096-token context), with lengths that are no
multiple of a tile in between.  Queries, keys and values are N(0,1).  Masks come from scores with the
structure of averaged attention (a band, sink columns, strided columns, sampling noise of the
calibration set) through the library's own selection, whose result depends on the scores alone.
"""
from __future__ import annotations

import math

import torch

import paper_2012_02030_b200.binding as ap

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _case(name, op, B, H, Lq, Lk, d, dtype, causal, keep, diag=True, rule="head", bias=True, height=3.0, width=16.0,
          sinks=8, stride=0, samples=1024):
    """One case.  height, width, sinks, stride, samples: band, sink columns and strided columns of the
    averaged attention, and the number of calibration sequences behind it (its noise)."""
    c = dict(op=op, B=B, H=H, Lq=Lq, Lk=Lk, d=d, dtype=dtype, causal=causal, keep=keep, diag=diag, rule=rule,
             bias=bias, height=height, width=width, sinks=sinks, stride=stride, samples=samples)
    return dict(c, name=name) if name else c


def listed():
    bert = dict(height=2.0, width=10.0, sinks=0, samples=2048)
    long = dict(height=3.0, width=64.0, sinks=16, stride=256, samples=64)
    return [
        # the smallest call: a toy model in fp32, two sequences and two heads
        _case("fwd_tiny_f32", "fwd", 2, 2, 128, 128, 64, "f32", False, 0.10, height=3.0, width=8.0, sinks=4, samples=32),
        # encoder of a BERT-base-shaped classifier, a batch of 32 sequences of 128: many short rows, launch-bound
        _case("fwd_bert", "fwd", 32, 12, 128, 128, 64, "bf16", False, 0.50, **bert),
        # language model with memory keys, half precision, segment and memory lengths that are no multiple of 16
        _case("fwd_memory_ragged_f16", "fwd", 16, 16, 375, 759, 64, "f16", True, 0.10, height=3.0, width=32.0, sinks=8,
              samples=256),
        # 4096-token causal context, the shape that the pruned forward is for
        _case("fwd_long", "fwd", 4, 16, 4096, 4096, 128, "bf16", True, 0.05, **long),
        # the same shape unpruned: what the pruned forward is compared with, and the largest contraction
        _case("dense_long", "dense", 4, 16, 4096, 4096, 128, "bf16", True, 1.0, **long),
        # retraining of a translation model's cross-attention: ragged source and target lengths
        _case("train_cross_ragged", "train", 64, 8, 250, 231, 64, "bf16", False, 0.50, diag=False, height=2.0, width=12.0,
              sinks=0, samples=4096),
        # retraining at the long context
        _case("train_long", "train", 4, 16, 4096, 4096, 128, "bf16", True, 0.05, **long),
        # calibration of a language model, segments of 512
        _case("accumulate_lm", "accumulate", 16, 16, 512, 512, 64, "bf16", True, 0.10),
        # calibration at the long context
        _case("accumulate_long", "accumulate", 4, 16, 4096, 4096, 128, "bf16", True, 0.05, **long),
        # pruning one layer of the language model with the paper's rule (one threshold for the layer)
        _case("mask_lm_layer", "mask", 16, 16, 512, 512, 64, "bf16", True, 0.10, rule="layer"),
        # pruning at the long context, one threshold per head
        _case("mask_long", "mask", 4, 16, 4096, 4096, 128, "bf16", True, 0.05, **long),
        # language model normalised by 1.5-entmax
        _case("entmax_lm", "entmax", 16, 16, 512, 512, 64, "bf16", True, 0.10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _domain(c):
    """Entries of one head that are neither pruned by causality nor outside the matrix."""
    if c["causal"]:
        return c["Lq"] * (c["Lq"] + 1) // 2 + c["Lq"] * (c["Lk"] - c["Lq"])
    return c["Lq"] * c["Lk"]


def draw(rng):
    op = rng.choice(["fwd", "fwd", "fwd", "dense", "train", "train", "accumulate", "accumulate", "mask", "mask", "entmax"])
    dtype = "bf16" if op in ("train", "mask", "entmax") and rng.random() < 0.7 else rng.choice(["bf16", "bf16", "bf16", "f16", "f32"])
    if dtype == "f32" and op not in ("fwd", "accumulate"):
        dtype = "f16"
    d = rng.choice([64, 64, 128])
    H = rng.choice([2, 4, 8, 12, 16, 32])
    # what the largest listed case of the kind computes, in multiply-adds of one contraction: fp32 runs
    # on the CUDA cores and only toy models use it; entmax is listed at the language model's shape
    most = 4 * 16 * (4096 * 4097 // 2) * 128
    most = most // 256 if dtype == "f32" else most // 8 if op == "entmax" else most // 3 if op == "train" else most
    hi = 512 if dtype == "f32" else 1024 if op == "entmax" else 4096
    form = rng.choice(["self", "causal", "causal", "memory", "cross"])
    while True:
        Lq = _log(rng, 64, hi)
        if rng.random() < 0.4:
            Lq = -(-Lq // 64) * 64
        Lk = Lq
        if form == "memory":
            Lk = min(hi, Lq + rng.choice([Lq, _log(rng, 16, hi)]))
        elif form == "cross":
            Lk = max(48, min(hi, int(Lq * rng.uniform(0.5, 2.0))))
        c = _case(None, op, 1, H, Lq, Lk, d, dtype, form in ("causal", "memory"), 1.0, bias=True)
        if H * _domain(c) * d <= most and H * Lq * Lk <= 16 * 4096 * 4096:
            break
        H = max(1, H // 2)
    c["B"] = max(1, min(_log(rng, 1, 64), most // (H * _domain(c) * d)))
    c["H"] = H
    c["keep"] = 1.0 if op == "dense" else round(math.exp(rng.uniform(math.log(0.05), math.log(0.5))), 3)
    c["diag"] = form != "cross"
    c["rule"] = rng.choice(["head", "head", "layer"])
    c["bias"] = rng.random() < 0.7
    c["height"] = round(rng.uniform(2.0, 3.0), 2)
    c["width"] = round(math.exp(rng.uniform(math.log(8.0), math.log(64.0))), 1)
    c["sinks"] = rng.choice([0, 4, 8, 16])
    c["stride"] = 256 if Lk >= 1024 and rng.random() < 0.5 else 0
    c["samples"] = _log(rng, 64, 4096)
    return c


def _bias(c, h, i, j):
    """Additive bias of head h on the scaled logits (the structure of trained attention)."""
    off = c["Lk"] - c["Lq"]
    if c["causal"]:
        dist = (i + off - j).clamp(min=0.0)
    else:
        dist = (i * (c["Lk"] / c["Lq"]) - j).abs()
    b = c["height"] * torch.exp(-dist / (c["width"] * (1.0 + h / (2.0 * c["H"]))))
    if c["sinks"]:
        b = b + 2.0 * (j < c["sinks"])
    if c["stride"]:
        b = b + 1.5 * (torch.remainder(j, c["stride"]) == 0)
    return b


def _positions(c):
    i = torch.arange(c["Lq"], dtype=torch.float32, device="cuda").view(-1, 1)
    j = torch.arange(c["Lk"], dtype=torch.float32, device="cuda").view(1, -1)
    return i, j, (j <= i + (c["Lk"] - c["Lq"])) if c["causal"] else None


def _scores(c, g):
    """Averaged attention [H,Lq,Lk]: exp(bias) with the noise that averaging exp(N(0,1)) over the
    calibration sequences leaves (same mean and variance, log-normal), each row divided by its sum."""
    out = torch.empty((c["H"], c["Lq"], c["Lk"]), dtype=torch.float32, device="cuda")
    sigma = math.sqrt(math.log1p((math.e - 1.0) / c["samples"]))
    i, j, domain = _positions(c)
    for h in range(c["H"]):
        s = torch.randn((c["Lq"], c["Lk"]), generator=g, dtype=torch.float32, device="cuda")
        s = torch.exp(s.mul_(sigma).add_(_bias(c, h, i, j)))
        if domain is not None:
            s *= domain
        torch.div(s, s.sum(dim=1, keepdim=True), out=out[h])
    return out


def _select(c, s, out):
    """The selection of one case into the buffers of `out`."""
    fn = ap.ap_build_mask_layer if c["rule"] == "layer" else ap.ap_build_mask
    fn(s, c["keep"], causal=c["causal"], keep_diag=c["diag"], mask=out["mask"], tiles=out["tiles"],
       nnz_per_head=out["nnz"], workspace=out["workspace"])


def prepare(case, seed):
    c = case
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 17)
    B, H, Lq, Lk, d, dt = c["B"], c["H"], c["Lq"], c["Lk"], c["d"], DTYPES[c["dtype"]]

    def randn(L):
        return torch.randn((B, H, L, d), generator=g, dtype=torch.float32, device="cuda").to(dt)

    s = dict(case=c)
    if c["op"] == "accumulate":
        s.update(acc=torch.zeros((H, Lq, Lk), dtype=torch.float32, device="cuda"), Q=randn(Lq), K=randn(Lk), bias=None)
        if c["bias"]:
            i, j, domain = _positions(c)
            s["bias"] = torch.stack([_bias(c, h, i, j) if domain is None else _bias(c, h, i, j) * domain for h in range(H)])
        return s
    s["tiles"] = ap.Tiles(H, Lq, Lk)
    if c["op"] == "dense":
        ap.ap_dense_tiles(s["tiles"], causal=c["causal"])
    else:
        s.update(mask=torch.zeros((H, Lq, Lk), dtype=torch.uint8, device="cuda"),
                 nnz=torch.zeros(H, dtype=torch.int64, device="cuda"),
                 workspace=torch.empty(ap.ap_build_mask_workspace_bytes(H, Lq, Lk), dtype=torch.uint8, device="cuda"))
        scores = _scores(c, g)
        if c["op"] == "mask":
            s["scores"] = scores
            return s
        _select(c, scores, s)
        del s["mask"], s["workspace"]
    s.update(Q=randn(Lq), K=randn(Lk), V=randn(Lk))
    if c["op"] == "train":
        s["dO"] = randn(Lq)
    return s


def run(state):
    s, c = state, state["case"]
    op = c["op"]
    if op == "accumulate":
        ap.ap_accumulate_attention(s["acc"], s["Q"], s["K"], bias=s["bias"], causal=c["causal"])
        return s["acc"]
    if op == "mask":
        _select(c, s["scores"], s)
        t = s["tiles"]
        return dict(mask=s["mask"], nnz=s["nnz"], row_ptr=t.row_ptr, col_idx=t.col_idx, flags=t.flags, bitmap=t.bitmap,
                    groups=t.groups, round_ptr=t.round_ptr, round_rows=t.round_rows, round_info=t.round_info,
                    round_bitmap=t.round_bitmap)
    if op == "entmax":
        return ap.ap_sparse_attention_entmax15_fwd(s["Q"], s["K"], s["V"], s["tiles"])
    O = ap.ap_sparse_attention_fwd(s["Q"], s["K"], s["V"], s["tiles"])
    if op != "train":
        return O
    dQ, dK, dV = ap.ap_sparse_attention_bwd(s["Q"], s["K"], s["V"], O, s["dO"], s["tiles"])
    return dict(O=O, dQ=dQ, dK=dK, dV=dV)


def work(case):
    c = case
    B, H, Lq, Lk, d = c["B"], c["H"], c["Lq"], c["Lk"], c["d"]
    e = 4 if c["dtype"] == "f32" else 2
    n = _domain(c)
    kept = max(Lq if c["diag"] and (c["causal"] or Lq == Lk) else 0, min(n, int(c["keep"] * n + 0.5)))
    q, k = B * H * Lq * d * e, B * H * Lk * d * e
    bits = 0 if c["op"] == "dense" else H * n // 8
    if c["op"] == "accumulate":  # Q, K, the sum read and written, the bias; one contraction
        return {"bytes": q + k + (12 if c["bias"] else 8) * H * n, "flops": 2 * d * B * H * n}
    if c["op"] == "mask":  # the scores once; the mask as bytes and as bits
        return {"bytes": 4 * H * n + H * Lq * Lk + bits, "flops": 0}
    if c["op"] == "train":  # forward: Q K V -> O; backward: Q K V O dO -> dQ dK dV, five contractions
        return {"bytes": 6 * q + 6 * k + 2 * bits, "flops": 14 * d * B * H * kept}
    return {"bytes": 2 * q + 2 * k + bits, "flops": 4 * d * B * H * kept}


def tolerance(case):
    """Masks and lists are whole numbers.  Sums of softmax weights are fp32.  Attention outputs are rounded to
    the 16-bit type once, the weights before them once as well (2^-9 and 2^-12 each); gradients pass
    through two more roundings (P, dS) and the rounded O."""
    if case["op"] == "mask":
        return "exact"
    if case["op"] == "accumulate":
        return {"rel": 2e-5}
    if case["dtype"] == "f32":
        return {"rel": 1e-5}
    if case["op"] == "train":
        return {"rel": 1e-2 if case["dtype"] == "bf16" else 2e-3}
    return {"rel": 5e-3 if case["dtype"] == "bf16" else 1e-3}
