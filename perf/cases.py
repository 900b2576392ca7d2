"""The work that users of this library have it do, as cases that can be timed and compared.

Three kinds of call, each through the public entry points of `paper_2609_33916_b200`:

  attention   softmax attention over whole sequences: forward and backward in one call ("fused", the training step of the
              benchmark configurations), forward then backward as two calls ("separate", what an autograd function does), or
              forward alone ("forward", the prefill of a prompt)
  decode      one new query per head over a cache of keys and values
  block       forward and backward of a whole pre-norm transformer block (RMSNorm, packed projection, attention, output
              projection, gated MLP), the composition in `paper_2609_33916_b200/block.py`

`prepare` makes what a user's program holds before the call (tensors, descriptor, workspace); `run` is one pass.
Inputs are i.i.d. N(0,1) (weights scaled by their fan-in, gains around one), like those of the tests and the benchmark.
"""
import math

import torch

from paper_2609_33916_b200 import binding as mb
from paper_2609_33916_b200.block import TransformerBlock


def _attention(name, call, dtype, B, H, Hkv, n, d, causal, tokens=False):
    return {"name": name, "kind": "attention", "call": call, "dtype": dtype, "B": B, "H": H, "Hkv": Hkv, "n": n, "d": d,
            "causal": causal, "tokens": tokens}


def _decode(name, dtype, B, H, Hkv, n, d):
    return {"name": name, "kind": "decode", "dtype": dtype, "B": B, "H": H, "Hkv": Hkv, "n": n, "d": d}


def _block(name, B, n, H, d, d_ff, causal):
    return {"name": name, "kind": "block", "B": B, "n": n, "H": H, "d": d, "d_ff": d_ff, "causal": causal}


def listed():
    return [
        # configuration 1, fp32: the smallest training step, all launch latency (unit tests, gradient checks, toy models)
        _attention("f32_tiny", "fused", "f32", 1, 1, 1, 128, 64, False),
        # fp32 at the shape of the paper's own GPU tables (two sequences, one head): research code that wants full precision
        _attention("f32_paper_n2048", "fused", "f32", 2, 1, 1, 2048, 64, False),
        # configuration 2: a small encoder's training step, 64-column heads
        _attention("train_small_d64", "fused", "bf16", 4, 8, 8, 1024, 64, False),
        # configuration 5's shortest sequence: short causal sequences, many heads
        _attention("train_short_causal", "fused", "bf16", 1, 32, 32, 512, 128, True),
        # configuration 3: the ordinary causal training step
        _attention("train_mid_causal", "fused", "bf16", 2, 16, 16, 4096, 128, True),
        # configuration 4, the default of bench.py: a long sequence, the largest case
        _attention("train_long", "fused", "bf16", 1, 16, 16, 16384, 128, False),
        # forward and backward as two calls on token-major tensors with shared K/V heads, a ragged length and a wide head
        _attention("train_wide_gqa_ragged", "separate", "bf16", 1, 16, 4, 3001, 192, True, tokens=True),
        # prefill of one long prompt with shared K/V heads, forward only
        _attention("prefill_gqa", "forward", "bf16", 1, 32, 8, 5000, 128, True, tokens=True),
        # one decoding step of a single short conversation: latency
        _decode("decode_short", "bf16", 1, 16, 16, 1000, 64),
        # one decoding step of a batch over long caches with grouped heads: 1.07 GB read
        _decode("decode_gqa_long", "bf16", 8, 32, 8, 32768, 128),
        # a block at the paper's traffic-check size: a toy model's step, all launches
        _block("block_tiny", 2, 256, 1, 64, 256, False),
        # a model-sized block around configuration 3's attention
        _block("block_mid_causal", 2, 4096, 16, 128, 8192, True),
    ]


# No drawn case costs more than the largest listed ones: model flops of an attention pass, bytes of a cache, block flops.
_MOST_BF16 = 14.0 * 16 * 16384.0 ** 2 * 128
_MOST_F32 = 4e10
_MOST_CACHE = 8 * 8 * 32768 * 128 * 2 * 2
_MOST_BLOCK = 4.0e12


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: attention (half of the draws), decode and block (a quarter each)."""
    kind = rng.choice(("attention", "attention", "decode", "block"))
    while True:
        if kind == "attention":
            call, causal = rng.choice(("fused", "fused", "separate", "forward")), rng.random() < 0.6
            if rng.random() < 0.2:
                H = rng.choice((1, 2, 4, 8))
                c = _attention("", call, "f32", rng.choice((1, 2)), H, H, _log(rng, 64, 2048), rng.choice((64, 128)), causal)
            else:
                H = rng.choice((8, 16, 32))
                c = _attention("", call, "bf16", rng.choice((1, 2, 4)), H, H // rng.choice((1, 1, 4, 8)), _log(rng, 128, 16384),
                               rng.choice((64, 64, 128, 128, 128, 80, 96, 192, 256)), causal, rng.random() < 0.5)
            # head sizes other than 128 run at a lower rate per model flop: half the flops cost about as much
            most = _MOST_F32 if c["dtype"] == "f32" else _MOST_BF16 if c["d"] == 128 else _MOST_BF16 / 2
            if _flops_attention(dict(c, call="fused")) > most:
                continue
        elif kind == "decode":
            H = rng.choice((8, 16, 32))
            c = _decode("", rng.choice(("bf16", "bf16", "bf16", "f32")), _log(rng, 1, 32), H, H // rng.choice((1, 2, 4, 8)),
                        _log(rng, 256, 32768), rng.choice((64, 128)))
            if _bytes_cache(c) > _MOST_CACHE:
                continue
        else:
            H, d = rng.choice((1, 2, 4, 8, 16)), rng.choice((64, 128))
            d_ff = rng.choice((4 * H * d, 8 * (H * d // 3)))
            c = _block("", rng.choice((1, 2)), _log(rng, 128, 4096), H, d, d_ff, rng.random() < 0.6)
            if work(c)["flops"] > _MOST_BLOCK:
                continue
        del c["name"]
        return c


def _randn(gen, dtype, *shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).to(dtype)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    state = {"case": case}
    if case["kind"] == "block":
        B, n, dm, ff = case["B"], case["n"], case["H"] * case["d"], case["d_ff"]
        bf = torch.bfloat16
        block = TransformerBlock(torch, B, n, case["H"], case["d"], ff, case["causal"])
        w = {k: _randn(gen, bf, dm, dm) * dm ** -0.5 for k in ("Wq", "Wk", "Wv", "Wo")}
        w.update(W1=_randn(gen, bf, ff, dm) * dm ** -0.5, W3=_randn(gen, bf, ff, dm) * dm ** -0.5,
                 W2=_randn(gen, bf, dm, ff) * ff ** -0.5)
        w.update({k: 1 + 0.25 * _randn(gen, bf, dm) for k in ("g1", "g2")})
        state.update(block=block, w=block.prepare_weights(w), x=_randn(gen, bf, B * n, dm), dy=_randn(gen, bf, B * n, dm))
        return state
    B, H, Hkv, n, d = (case[k] for k in ("B", "H", "Hkv", "n", "d"))
    dtype, code = (torch.float32, mb.MOA_F32) if case["dtype"] == "f32" else (torch.bfloat16, mb.MOA_BF16)
    if case["kind"] == "decode":
        state["desc"] = mb.make_decode_desc(B, H, n, d, d ** -0.5, code, H_kv=Hkv)
        state.update(q=_randn(gen, dtype, B, H, d), K=_randn(gen, dtype, B, Hkv, n, d), V=_randn(gen, dtype, B, Hkv, n, d))
        state.update(out=torch.empty_like(state["q"]), lse=torch.empty((B, H), dtype=torch.float32, device="cuda"))
        need = mb.moa_decode_workspace_bytes(state["desc"])
    else:
        shape = (lambda heads: (B, n, heads, d)) if case["tokens"] else (lambda heads: (B, heads, n, d))
        state["desc"] = mb.make_desc(B, H, n, d, case["causal"], d ** -0.5, dtype=code, H_kv=Hkv,
                                     layout=mb.MOA_LAYOUT_BNHD if case["tokens"] else mb.MOA_LAYOUT_BHND)
        state.update(Q=_randn(gen, dtype, *shape(H)), K=_randn(gen, dtype, *shape(Hkv)), V=_randn(gen, dtype, *shape(Hkv)))
        state.update(O=torch.empty_like(state["Q"]), L=torch.empty((B, H, n), dtype=torch.float32, device="cuda"))
        op = {"fused": mb.MOA_OP_FUSED, "separate": mb.MOA_OP_BWD, "forward": mb.MOA_OP_FWD}[case["call"]]
        if case["call"] != "forward":
            state["dO"] = _randn(gen, dtype, *shape(H))
            state.update(dQ=torch.empty_like(state["Q"]), dK=torch.empty_like(state["K"]), dV=torch.empty_like(state["V"]))
        need = mb.moa_attn_workspace_bytes(state["desc"], op)
    state["ws"] = torch.empty(max(16, need), dtype=torch.uint8, device="cuda")
    return state


def run(s):
    case = s["case"]
    if case["kind"] == "block":
        y = s["block"].forward(s["x"], s["w"])
        dx, grads = s["block"].backward(s["x"], s["w"], s["dy"])
        return {"y": y, "dx": dx, **{"d" + k: v for k, v in grads.items()}}
    if case["kind"] == "decode":
        mb.moa_decode_attn(s["desc"], s["q"], s["K"], s["V"], s["out"], s["lse"], s["ws"])
        return {"out": s["out"], "lse": s["lse"]}
    if case["call"] == "fused":
        mb.moa_attn_fused_fwd_bwd(s["desc"], s["Q"], s["K"], s["V"], s["dO"], s["O"], s["L"], s["dQ"], s["dK"], s["dV"], s["ws"])
    else:
        mb.moa_attn_fwd(s["desc"], s["Q"], s["K"], s["V"], s["O"], s["L"])
        if case["call"] == "separate":
            mb.moa_attn_bwd(s["desc"], s["Q"], s["K"], s["V"], s["O"], s["L"], s["dO"], s["dQ"], s["dK"], s["dV"], s["ws"])
    return {k: s[k] for k in ("O", "L", "dQ", "dK", "dV") if k in s}


def _flops_attention(case):
    n = case["n"]
    pairs = case["B"] * case["H"] * (n * (n + 1) / 2 if case["causal"] else float(n) ** 2)
    return (4.0 if case["call"] == "forward" else 14.0) * pairs * case["d"]


def _bytes_cache(case):
    return 2.0 * case["B"] * case["Hkv"] * case["n"] * case["d"] * (4 if case["dtype"] == "f32" else 2)


def work(case):
    """Model flops (two products forward, five backward) and every input read and output written once."""
    B, H, n, d = (case[k] for k in ("B", "H", "n", "d"))
    if case["kind"] == "block":
        T, dm, ff = B * n, H * d, case["d_ff"]
        att = _flops_attention(dict(case, call="fused"))
        return {"flops": 24.0 * T * dm * dm + 18.0 * T * dm * ff + att,
                "bytes": 2.0 * (4 * T * dm + 2 * (4 * dm * dm + 3 * dm * ff + 2 * dm))}
    size = 4 if case["dtype"] == "f32" else 2
    if case["kind"] == "decode":
        return {"flops": 4.0 * B * H * n * d, "bytes": _bytes_cache(case) + B * H * (2.0 * d * size + 4)}
    queries, keys = B * H * n * d, B * case["Hkv"] * n * d
    arrays = 2 * queries + 2 * keys if case["call"] == "forward" else 4 * queries + 4 * keys      # Q K V O (dO dQ dK dV)
    return {"flops": _flops_attention(case), "bytes": float(arrays) * size + 4.0 * B * H * n}


def tolerance(case):
    """About four times what the library's results were off from the same definitions evaluated in 64 bits (2-norm ratios of the
    worst output; "max" for attention is set by gradients of causal rows that see few keys):
    fp32 9.7e-7 (largest element 1.5e-5); bf16 attention and decode 2.5e-3 (0.11); the block, whose bf16 stages compound,
    6.6e-3 (4.4e-2)."""
    if case["kind"] == "block":
        return {"rel": 2.5e-2, "max": 0.2}
    if case["dtype"] == "f32":
        return {"rel": 4e-6, "max": 6e-5}
    return {"rel": 1e-2, "max": 0.4 if case["kind"] == "attention" else 2e-2}
