"""What a program that serves long prompts has this library do: prefill layers (dense, packed, chunked), decode steps.

A case is one call sequence of one attention layer, through the functions of ``paper_2608_17336_b200.binding``:

  prefill  Q, K and V of a layer and its routing map are on the GPU; a pass quantises Q and K, packs the map and runs
           the fused kernel (with ``otf`` the quantiser runs inside it: no INT8 copies in device memory).
  varlen   the same over a packed batch of prompts of unequal lengths (token-major tensors, as a projection leaves them).
  chunk    the last ``L`` tokens of a ``ctx``-token context whose key cache (FP16 and INT8) and value cache (``v8``:
           INT8 with block scales, else FP16) are filled; a pass quantises the chunk's queries and keys and attends.
  decode   one new token per sequence over an INT8 key/value cache; ``ragged``: the sequences have unequal lengths.

Values are N(0,1), or have a few channels per head scaled by 8 (``outlier``), or heavy-tailed keys (``tails``), as
activations of such layers do.  Routing is drawn per tile group: INT8 with probability ``f8``; with ``band`` the groups
within 1024 tokens of the diagonal stay FP16 and each head has a probability of its own; ``pin`` keeps the diagonal FP16.
"""
import math

import torch

from paper_2608_17336_b200 import binding as tm

BAND = 1024          # tokens next to the diagonal that a banded map keeps FP16
MOST_FLOPS = 2.0e13  # of a drawn prefill: the largest listed one needs 3.5e13


def _prefill(name, B, Hq, Hk, L, d, G, f8, values="normal", band=False, pin=False, lse=False, otf=False, half=False):
    return dict(name=name, kind="prefill", B=B, Hq=Hq, Hk=Hk, L=L, d=d, G=G, f8=f8, values=values, band=band, pin=pin,
                lse=lse, otf=otf, half=half)


def listed():
    return [
        # the smallest call: one short head of a small model; launches and latency count
        _prefill("prefill_1k_one_head_d64", 1, 1, 1, 1024, 64, 1, 0.5),
        # one Llama-style layer over an 8K prompt, activations with outlier channels, half of the groups INT8
        _prefill("prefill_8k_outliers", 1, 32, 32, 8192, 128, 1, 0.5, values="outlier"),
        # a batch of medium prompts, FP16 near the diagonal and a share of INT8 of its own for each head
        _prefill("prefill_8x4k_band", 8, 32, 32, 4096, 128, 2, 0.5, band=True),
        # the library's main workload: 32K tokens, 75 % INT8, diagonal pinned
        _prefill("prefill_32k", 1, 32, 32, 32768, 128, 4, 0.75, pin=True),
        # the longest context, heavy-tailed keys, 90 % INT8
        _prefill("prefill_128k_tails", 1, 8, 8, 131072, 128, 8, 0.9, values="tails"),
        # a batch on a model with 64-dimensional heads and grouped queries, ragged length, LSE wanted
        _prefill("prefill_4x2000_d64_gqa", 4, 32, 8, 2000, 64, 2, 0.5, lse=True),
        # a layer with grouped queries in the operand mode that keeps no INT8 copies in device memory
        _prefill("prefill_8k_on_the_fly", 1, 32, 8, 8192, 128, 2, 0.75, pin=True, otf=True),
        # continuous batching: sixteen prompts of 40 to 5000 tokens packed without padding
        dict(name="varlen_16_prompts", kind="varlen", n=16, shortest=40, longest=5000, Hq=32, Hk=8, d=128, G=2, f8=0.5,
             lens=7),
        # chunked prefill late in a long context, INT8 value cache
        dict(name="chunk_2k_of_24k_v8", kind="chunk", B=1, Hq=32, Hk=8, L=2048, ctx=24576, d=128, G=4, f8=0.75, v8=True,
             half=False),
        # a decode step of eight long sequences of one length, grouped queries
        dict(name="decode_8x32k", kind="decode", B=8, Hq=32, Hk=8, d=128, tile=128, max_len=32768, G=4, f8=0.75,
             ragged=False, splits=0, lens=0),
        # a decode step of a batch in mixed stages, splits left to the kernel
        dict(name="decode_16_ragged", kind="decode", B=16, Hq=32, Hk=8, d=128, tile=128, max_len=12288, G=2, f8=0.75,
             ragged=True, splits=-1, lens=3),
        # the same on a model with 64-dimensional heads
        dict(name="decode_16x8k_d64", kind="decode", B=16, Hq=32, Hk=8, d=64, tile=64, max_len=8192, G=4, f8=0.75,
             ragged=True, splits=0, lens=5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["prefill"] * 6 + ["varlen"] * 2 + ["chunk"] * 2 + ["decode"] * 4)
    f8 = rng.choice([0.0, 0.25, 0.5, 0.75, 0.9, 1.0])
    heads = rng.choice([(1, 1), (8, 8), (32, 32), (16, 16), (32, 8), (16, 4), (28, 4), (64, 8)])
    G = rng.choice([1, 2, 4, 8])
    while True:
        if kind == "prefill":
            d = rng.choice([128, 128, 128, 64])
            c = _prefill("", rng.choice([1, 1, 2, 4, 8]), *heads, _log(rng, 100, 60000), d, G, f8,
                         values=rng.choice(["normal", "outlier", "tails"]), band=rng.random() < 0.3, pin=rng.random() < 0.5,
                         lse=rng.random() < 0.3, otf=d == 128 and rng.random() < 0.15, half=rng.random() < 0.2)
            if c["otf"]:
                c["half"] = False
        elif kind == "varlen":
            c = dict(kind="varlen", n=rng.randint(2, 48), shortest=rng.randint(1, 200), longest=_log(rng, 300, 16000),
                     Hq=heads[0], Hk=heads[1], d=rng.choice([128, 128, 64]), G=G, f8=f8, lens=rng.randrange(1 << 20))
        elif kind == "chunk":
            L = _log(rng, 128, 8192)
            d = rng.choice([128, 128, 128, 64])
            c = dict(kind="chunk", B=rng.choice([1, 1, 2]), Hq=heads[0], Hk=heads[1], L=L, ctx=L + d * _log(rng, 1, 40000 // d),
                     d=d, G=G, f8=f8, v8=rng.random() < 0.5, half=rng.random() < 0.2)
        else:
            hk = rng.choice([1, 2, 4, 8, 32])
            d = rng.choice([128, 128, 64])
            c = dict(kind="decode", B=_log(rng, 1, 64), Hq=hk * rng.choice([1, 2, 4, 8]), Hk=hk, d=d,
                     tile=rng.choice([128, 128, 64]) if d == 128 else rng.choice([64, 128]), max_len=_log(rng, 500, 70000),
                     G=G, f8=f8, ragged=rng.random() < 0.5, splits=rng.choice([0, 0, -1]), lens=rng.randrange(1 << 20))
        c.pop("name", None)
        w = work(c)
        if w["flops"] <= MOST_FLOPS and w["bytes"] <= 4e9:
            return c


# ------------------------------------------------------------------------------------------------------ sizes of a case

def _seq_lens(c):
    """Lengths of a packed batch or of the cached sequences: spread over their range, the same for every seed."""
    gen = torch.Generator().manual_seed(1000 + c["lens"])
    if c["kind"] == "varlen":
        u = torch.rand(c["n"], generator=gen)
        return [int(x) for x in torch.exp(math.log(c["shortest"]) + u * math.log(c["longest"] / c["shortest"])).ceil()]
    if not c["ragged"]:
        return [c["max_len"]] * c["B"]
    u = torch.rand(c["B"], generator=gen)
    return [max(1, int(c["max_len"] * float(x))) for x in u]


def work(c):
    """Each tensor that the caller hands over or gets back once; multiply-adds of the legal (query, key) pairs."""
    d, hq, hk = c["d"], c["Hq"], c["Hk"]
    if c["kind"] == "decode":
        n = sum(_seq_lens(c))
        return {"bytes": n * hk * d * (1.0 + c["f8"] + 2.0 * (1.0 - c["f8"])) + 4.0 * c["B"] * hq * d, "flops": 4.0 * n * hq * d}
    if c["kind"] == "varlen":
        lens = _seq_lens(c)
        rows, keys, pairs = sum(lens), sum(lens), sum(n * (n + 1) / 2 for n in lens)
    elif c["kind"] == "chunk":
        rows, keys = c["B"] * c["L"], c["B"] * c["ctx"]
        pairs = c["B"] * (c["L"] * (c["ctx"] - c["L"]) + c["L"] * (c["L"] + 1) / 2)
    else:
        rows = keys = c["B"] * c["L"]
        pairs = c["B"] * c["L"] * (c["L"] + 1) / 2
    # Q read and O written in FP16, K and V read (a chunk reads its key cache by route, and its values as they are cached)
    key_bytes = (1.0 * c["f8"] + 2.0 * (1.0 - c["f8"]) + (1.0 if c["v8"] else 2.0)) if c["kind"] == "chunk" else 4.0
    codes = 0.0 if c.get("otf") else 1.0 * d * (rows * hq + (rows if c["kind"] == "chunk" else keys) * hk)
    return {"bytes": 4.0 * rows * hq * d + key_bytes * keys * hk * d + codes, "flops": 4.0 * pairs * hq * d}


def tolerance(c):
    """Probabilities and outputs are rounded to FP16, sums are FP32; INT8 codes, scales and mask words are exact.  Against
    the definition in float64 (on the same codes) the outputs of all kinds of case differ by 2.4e-4 to 3.7e-4 (2-norm) and
    by at most 3.8e-3 of the root mean square; four times that is allowed."""
    return {"rel": 1.4e-3, "max": 1.5e-2, "differ": 0.0}


# ------------------------------------------------------------------------------------------------------ inputs

def _values(gen, shape, recipe, head_axis, keys=False):
    x = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float16)
    if recipe == "outlier":
        h, d = shape[head_axis], shape[-1]
        ch = (torch.arange(4, device="cuda")[None, :] * 29 + torch.arange(h, device="cuda")[:, None] * 7) % d
        gain = torch.ones((h, d), device="cuda", dtype=torch.float16).scatter_(1, ch, 8.0)
        x *= gain.view([1] * head_axis + [h] + [1] * (len(shape) - head_axis - 2) + [d])
    elif recipe == "tails" and keys:
        # Student-t with three degrees of freedom
        chi = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float16).square_()
        for _ in range(2):
            chi += torch.randn(shape, generator=gen, device="cuda", dtype=torch.float16).square_()
        x = (x / (chi / 3.0).sqrt_().clamp_(min=1e-2)).clamp_(-500.0, 500.0)
    return x


def _route(gen, rows, groups, Hk, tile, G, f8, band=False):
    """uint8 [1, Hk, rows, groups]; the packer ignores what lies above the diagonal."""
    u = torch.rand((1, Hk, rows, groups), generator=gen, device="cuda")
    if not band:
        return (u < f8).to(torch.uint8)
    p = torch.rand((1, Hk, 1, 1), generator=gen, device="cuda")
    first = torch.arange(rows, device="cuda")[:, None] * tile
    last = (torch.arange(groups, device="cuda")[None, :] + 1) * (G * tile) - 1
    return ((u < p) & (first - last >= BAND)).to(torch.uint8)


def _bits_to_words(bits):
    """bool [..., T_mask] -> int32-typed words [..., W], bit g of word g / 32."""
    t = bits.shape[-1]
    w = -(-t // 32)
    padded = torch.zeros(bits.shape[:-1] + (w * 32,), dtype=torch.int64, device=bits.device)
    padded[..., :t] = bits.to(torch.int64)
    words = (padded.view(bits.shape[:-1] + (w, 32)) << torch.arange(32, device=bits.device)).sum(-1)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32).contiguous()


def prepare(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return {"prefill": _prepare_prefill, "varlen": _prepare_varlen, "chunk": _prepare_chunk, "decode": _prepare_decode}[c["kind"]](c, gen)


def _prepare_prefill(c, gen):
    B, Hq, Hk, L, d, G, tile = c["B"], c["Hq"], c["Hk"], c["L"], c["d"], c["G"], c["d"]
    p = tm.problem(B, Hq, Hk, L, d, tile, tile, G, quant_blk_k=tile // 2 if c["half"] else 0,
                   flags=tm.QUANT_ON_THE_FLY if c["otf"] else 0)
    q, k, v = (_values(gen, (B, h, L, d), c["values"] if name != "v" else "normal", 1, name == "k")
               for name, h in (("q", Hq), ("k", Hk), ("v", Hk)))
    return dict(run=_run_prefill, p=p, q=q, k=k, v=v, route=_route(gen, p.T_m, p.T_mask, Hk, tile, G, c["f8"], c["band"]),
                pin=c["pin"], lse=c["lse"], otf=c["otf"],
                work=torch.empty(tm.tilemix_workspace_size(p), dtype=torch.uint8, device="cuda"))


def _run_prefill(s):
    p, q, k = s["p"], s["q"], s["k"]
    codes = (None,) * 4 if s["otf"] else tm.tilemix_quantize_qk(p, q, k)
    words, counts = tm.tilemix_pack_routing_mask(p, s["route"], s["pin"])
    r = tm.tilemix_attention_fwd(p, q, k, s["v"], *codes, words, want_lse=s["lse"], workspace=s["work"])
    return {"out": r["out"], "lse": r["lse"], "codes": list(codes), "words": words, "counts": counts}


def _prepare_varlen(c, gen):
    Hq, Hk, d, G, tile = c["Hq"], c["Hk"], c["d"], c["G"], c["d"]
    cu = [0]
    for n in _seq_lens(c):
        cu.append(cu[-1] + n)
    p = tm.problem(1, Hq, Hk, cu[-1], d, tile, tile, G)
    vl = tm.Varlen(cu)
    n = tm.tilemix_varlen_counts(p, vl)
    q, k, v = (torch.randn((cu[-1], h, d), generator=gen, device="cuda", dtype=torch.float16) for h in (Hq, Hk, Hk))
    route = (torch.rand((Hk, n["sum_T_m"], n["T_mask_max"]), generator=gen, device="cuda") < c["f8"]).to(torch.uint8)
    return dict(run=_run_varlen, p=p, vl=vl, q=q, k=k, v=v, route=route,
                work=torch.empty(tm.tilemix_varlen_workspace_size(p, vl), dtype=torch.uint8, device="cuda"))


def _run_varlen(s):
    p, vl, ws = s["p"], s["vl"], s["work"]
    codes = tm.tilemix_quantize_qk_varlen(p, vl, s["q"], s["k"], workspace=ws)
    words, counts = tm.tilemix_pack_routing_mask_varlen(p, vl, s["route"], workspace=ws)
    r = tm.tilemix_attention_fwd_varlen(p, vl, s["q"], s["k"], s["v"], *codes, words, workspace=ws)
    return {"out": r["out"], "codes": list(codes), "words": words, "counts": counts}


def _prepare_chunk(c, gen):
    B, Hq, Hk, L, ctx, d, G, tile = c["B"], c["Hq"], c["Hk"], c["L"], c["ctx"], c["d"], c["G"], c["d"]
    blk = tile // 2 if c["half"] else 0
    whole = tm.problem(B, Hk, Hk, ctx, d, tile, tile, G, quant_blk_q=blk, quant_blk_k=blk)
    p = tm.problem(B, Hq, Hk, L, d, tile, tile, G, quant_blk_k=blk)
    q = torch.randn((B, Hq, L, d), generator=gen, device="cuda", dtype=torch.float16)
    k, v = (torch.randn((B, Hk, ctx, d), generator=gen, device="cuda", dtype=torch.float16) for _ in range(2))
    _, k8, _, ks = tm.tilemix_quantize_qk(whole, k, k)
    words, _ = tm.tilemix_pack_routing_mask(whole, _route(gen, whole.T_m, whole.T_mask, Hk, tile, G, c["f8"]), True)
    s = dict(run=_run_chunk, p=p, ctx=ctx, q=q, k=k, k8=k8, ks=ks, words=words, v=v, v8=None, vs=None)
    if c["v8"]:
        s["v"] = None
        _, s["v8"], _, s["vs"] = tm.tilemix_quantize_qk(tm.problem(B, Hk, Hk, ctx, d, tile, tile, G), v, v)
        size = tm.tilemix_chunk_v8_workspace_size(p, ctx)
    else:
        size = tm.tilemix_workspace_size(p)
    s["work"] = torch.empty(size, dtype=torch.uint8, device="cuda")
    return s


def _run_chunk(s):
    # (the codes of the chunk's keys go into the key cache, which holds them here already)
    p, ctx, q, k = s["p"], s["ctx"], s["q"], s["k"]
    q8, k8_new, qs, ks_new = tm.tilemix_quantize_qk(p, q, k[:, :, ctx - p.seqlen:])
    if s["v8"] is not None:
        r = tm.tilemix_attention_fwd_chunk_v8(p, ctx, q, k, s["v8"], s["vs"], q8, s["k8"], qs, s["ks"], s["words"], workspace=s["work"])
    else:
        r = tm.tilemix_attention_fwd_chunk(p, ctx, q, k, s["v"], q8, s["k8"], qs, s["ks"], s["words"], workspace=s["work"])
    return {"out": r["out"], "codes": [q8, k8_new, qs, ks_new]}


def _prepare_decode(c, gen):
    B, Hq, Hk, d, tile, L, G = c["B"], c["Hq"], c["Hk"], c["d"], c["tile"], c["max_len"], c["G"]
    k, v = (torch.randn((B, Hk, L, d), generator=gen, device="cuda", dtype=torch.float16) for _ in range(2))
    k8, v8, ks, vs = tm.tilemix_quantize_qk(tm.problem(B, Hk, Hk, L, d, tile, tile, G), k, v)
    del v
    bits = torch.rand((1, Hk, -(-L // (G * tile))), generator=gen, device="cuda") < c["f8"]
    p = tm.decode_problem(B, Hq, Hk, d, L, tile, G, n_splits=c["splits"])
    return dict(run=_run_decode, p=p, q=torch.randn((B, Hq, d), generator=gen, device="cuda", dtype=torch.float16), k=k, k8=k8,
                ks=ks, v8=v8, vs=vs, words=_bits_to_words(bits),
                lens=torch.tensor(_seq_lens(c), dtype=torch.int32, device="cuda"),
                work=torch.empty(tm.tilemix_decode_workspace_size(p), dtype=torch.uint8, device="cuda"))


def _run_decode(s):
    r = tm.tilemix_decode_int8kv(s["p"], s["q"], s["k"], s["k8"], s["ks"], s["v8"], s["vs"], s["words"], s["lens"],
                                 want_lse=True, workspace=s["work"])
    return {"out": r["out"], "lse": r["lse"]}


def run(state):
    return state["run"](state)
