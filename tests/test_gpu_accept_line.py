"""The softmax steps' acceptance line: scores that climb from one 64-key step to the next by less than it, by about as much and by
more, so that steps are taken with a running maximum that lags, and redone.  Against float64 on the same codes."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("climb", [9.0, 14.5, 15.5, 21.5, 30.0])
@pytest.mark.parametrize("d,int8,v8", [(128, 0, False), (128, 1, False), (64, 0, False), (64, 1, False), (128, 1, True), (64, 0, True)])
def test_climbing_scores(d, int8, v8, climb):
    from paper_2608_17336_b200 import binding as tm
    B, Hq, Hk, L = 1, 2, 1, 520
    gen = torch.Generator(device=DEV).manual_seed(int(climb) + d)
    q, k, v = (torch.randn(s, generator=gen, device=DEV) for s in ((B, Hq, L, d), (B, Hk, L, d), (B, Hk, L, d)))
    q, k = 0.1 * q, 0.1 * k
    # channel 0 carries the climb: log2 of the score is 8 k0 log2(e) / sqrt(d); every row's maximum is at its own last keys
    q[..., 0] = 8.0
    k[..., 0] = (torch.arange(L, device=DEV) // 64) * climb * d ** 0.5 / (8.0 * 1.4426950408889634)
    if v8:
        v = v * 3000.0        # block scales near 100
    q, k, v = q.half(), k.half(), v.half()
    p = tm.problem(B, Hq, Hk, L, d, d, d, 1)
    q8, k8, qs, ks = tm.tilemix_quantize_qk(p, q, k)
    words, _ = tm.tilemix_pack_routing_mask(p, torch.full((1, Hk, p.T_m, p.T_mask), int8, dtype=torch.uint8, device=DEV))
    if v8:
        _, vc, _, vs = tm.tilemix_quantize_qk(tm.problem(B, Hk, Hk, L, d, d, d, 1), v, v)
        out = tm.tilemix_attention_fwd_chunk_v8(p, L, q, k, vc, vs, q8, k8, qs, ks, words)["out"]
        vd = vc.double() * vs.double().repeat_interleave(d, -1)[..., :L, None]
    else:
        out = tm.tilemix_attention_fwd(p, q, k, v, q8, k8, qs, ks, words)["out"]
        vd = v.double()
    rows = lambda s: s.double().repeat_interleave(d, -1)[..., :L, None]  # noqa: E731
    qd, kd = (q8.double() * rows(qs), k8.double() * rows(ks)) if int8 else (q.double(), k.double())
    s = (qd @ kd.expand(B, Hq, L, d).transpose(-1, -2)) / d ** 0.5
    s = s.masked_fill(torch.ones(L, L, dtype=torch.bool, device=DEV).triu(1), -torch.inf)
    ref = torch.softmax(s, -1) @ vd.expand(B, Hq, L, d)
    # a probability and an output are rounded to FP16 once each (2^-11 of at most the largest value behind a row); FP32 scores
    # of up to 2^9 carry 2^-15 each
    bound = (2.0 ** -10 + 2.0 ** -14) * vd.abs().amax()
    assert torch.isfinite(out).all()
    assert (out.double() - ref).abs().max() < bound


def _special_key_inputs(B, Hq, Hk, L, d, every, climb, v_top, seed):
    """One key in `every` carries the climb, the others score about 0: a step's row sum is that one probability."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    q, k, v = (torch.randn(s, generator=gen, device=DEV) for s in ((B, Hq, L, d), (B, Hk, L, d), (B, Hk, L, d)))
    q, k = 0.1 * q, 0.1 * k
    q[..., 0] = 8.0
    k[..., 0] = 0.0
    steps = torch.arange(0, L, every, device=DEV)
    k[:, :, steps, 0] = (steps // every) * climb * d ** 0.5 / (8.0 * 1.4426950408889634)
    if v_top:       # magnitudes between half and all of v_top, so that every block's scale is near v_top / 127
        v = torch.sign(v) * v_top * (0.5 + 0.5 * torch.rand(v.shape, generator=gen, device=DEV))
    return q.half(), k.half(), v.half()


def _reference(q, k, v, q8, k8, qs, ks, int8, blk_q, blk_k):
    """float64, one head pair after the other; q [Hq, L, d], v float64 [Hk, L, d]."""
    Hq, L, d = q.shape
    rep = Hq // k.shape[0]
    out = torch.empty((Hq, L, d), dtype=torch.float64, device=q.device)
    mask = torch.ones(L, L, dtype=torch.bool, device=q.device).triu(1)
    for h in range(Hq):
        g = h // rep
        if int8:
            qd = q8[h].double() * qs[h].double().repeat_interleave(blk_q)[:L, None]
            kd = k8[g].double() * ks[g].double().repeat_interleave(blk_k)[:L, None]
        else:
            qd, kd = q[h].double(), k[g].double()
        out[h] = torch.softmax((qd @ kd.T / d ** 0.5).masked_fill(mask, -torch.inf), -1) @ v[g]
    return out


# one tile per CTA, two adjacent tiles, the same rows of two heads
GRIDS = [(2, 1), (26, 26), (26, 13)]
# P of the key against the lagging maximum is 2^(climb - 6): below the line, and between it and what FP16 holds and beyond
CLIMBS = [20.7, 21.4, 22.2, 22.5, 22.8]


@pytest.mark.parametrize("climb", CLIMBS)
@pytest.mark.parametrize("Hq,Hk", GRIDS)
@pytest.mark.parametrize("d,form", [(128, "dense"), (128, "half"), (128, "otf"), (128, "varlen"), (64, "dense"), (64, "half"), (64, "varlen"),
                                    (64, "varlen half")])
def test_one_key_a_step(d, form, Hq, Hk, climb):
    from paper_2608_17336_b200 import binding as tm
    L = 520
    q, k, v = _special_key_inputs(1, Hq, Hk, L, d, 64, climb, 0.0, int(10 * climb) + d)
    blk_k = d // 2 if "half" in form else d
    for int8 in (0, 1):
        if "varlen" in form:
            cu = [0, L, L + 40]
            p, vl = tm.problem(1, Hq, Hk, cu[-1], d, d, d, 1, quant_blk_k=blk_k if "half" in form else 0), tm.Varlen(cu)
            n = tm.tilemix_varlen_counts(p, vl)
            ws = torch.empty(tm.tilemix_varlen_workspace_size(p, vl), dtype=torch.uint8, device=DEV)
            qt, kt, vt = (torch.cat([x[0].transpose(0, 1), x[0].transpose(0, 1)[:40]]).contiguous() for x in (q, k, v))
            codes = tm.tilemix_quantize_qk_varlen(p, vl, qt, kt, workspace=ws)
            route = torch.full((Hk, n["sum_T_m"], n["T_mask_max"]), int8, dtype=torch.uint8, device=DEV)
            words, _ = tm.tilemix_pack_routing_mask_varlen(p, vl, route, workspace=ws)
            out = tm.tilemix_attention_fwd_varlen(p, vl, qt, kt, vt, *codes, words, workspace=ws)["out"][:L].transpose(0, 1)
        else:
            p = tm.problem(1, Hq, Hk, L, d, d, d, 1, quant_blk_k=blk_k if form == "half" else 0, flags=tm.QUANT_ON_THE_FLY if form == "otf" else 0)
            codes = (None,) * 4 if form == "otf" else tm.tilemix_quantize_qk(p, q, k)
            words, _ = tm.tilemix_pack_routing_mask(p, torch.full((1, Hk, p.T_m, p.T_mask), int8, dtype=torch.uint8, device=DEV))
            out = tm.tilemix_attention_fwd(p, q, k, v, *codes, words)["out"][0]
        dense = tm.problem(1, Hq, Hk, L, d, d, d, 1, quant_blk_k=blk_k if "half" in form else 0)
        q8, k8, qs, ks = (x[0] for x in tm.tilemix_quantize_qk(dense, q, k))
        ref = _reference(q[0], k[0], v[0].double(), q8, k8, qs, ks, int8, d, blk_k)
        assert torch.isfinite(out).all()
        # (as above)
        assert (out.double() - ref).abs().max() < (2.0 ** -10 + 2.0 ** -14) * v.double().abs().amax(), int8


@pytest.mark.parametrize("climb", [13.1, 13.4, 13.9, 16.0])
@pytest.mark.parametrize("Hq,Hk", GRIDS)
@pytest.mark.parametrize("d,half", [(128, False), (128, True), (64, False), (64, True)])
def test_one_key_a_step_with_large_value_scales(d, half, Hq, Hk, climb):
    """An INT8 value cache whose block scales are near 480: the scaled probability has to fit FP16, not the probability."""
    from paper_2608_17336_b200 import binding as tm
    L = 520
    q, k, v = _special_key_inputs(1, Hq, Hk, L, d, 64, climb, 61000.0, int(10 * climb) + d)
    _, v8, _, vs = tm.tilemix_quantize_qk(tm.problem(1, Hk, Hk, L, d, d, d, 1), v, v)
    vd = v8[0].double() * vs[0].double().repeat_interleave(d, -1)[..., :L, None]
    blk_k = d // 2 if half else d
    for int8 in (0, 1):
        p = tm.problem(1, Hq, Hk, L, d, d, d, 1, quant_blk_k=blk_k if half else 0)
        codes = tm.tilemix_quantize_qk(p, q, k)
        words, _ = tm.tilemix_pack_routing_mask(p, torch.full((1, Hk, p.T_m, p.T_mask), int8, dtype=torch.uint8, device=DEV))
        out = tm.tilemix_attention_fwd_chunk_v8(p, L, q, k, v8, vs, codes[0], codes[1], codes[2], codes[3], words)["out"][0]
        ref = _reference(q[0], k[0], vd, *(x[0] for x in codes), int8, d, blk_k)
        assert torch.isfinite(out).all()
        assert (out.double() - ref).abs().max() < (2.0 ** -10 + 2.0 ** -14) * vd.abs().amax(), int8


@pytest.mark.parametrize("d,climb", [(128, 8.6), (128, 9.5), (64, 9.0)])
def test_a_rejected_step_moves_the_maximum(d, climb):
    """INT8 value cache, keys that stay `climb` binades above the first ones: 2^(climb - 6) a key is over the line of a step's
    sums.  If m stayed where it is, every step would be redone; that took 1.9 times as long, and takes as long as without."""
    from paper_2608_17336_b200 import binding as tm
    Hq, Hk, L, ctx = 32, 8, 1024, 8192
    gen = torch.Generator(device=DEV).manual_seed(d)
    whole, p = tm.problem(1, Hk, Hk, ctx, d, d, d, 1), tm.problem(1, Hq, Hk, L, d, d, d, 1)
    q, k, v = (0.1 * torch.randn(s, generator=gen, device=DEV) for s in ((1, Hq, L, d), (1, Hk, ctx, d), (1, Hk, ctx, d)))
    q[..., 0], k[..., 0] = 8.0, 0.0
    words, _ = tm.tilemix_pack_routing_mask(whole, torch.zeros((1, Hk, whole.T_m, whole.T_mask), dtype=torch.uint8, device=DEV))
    q, v = q.half(), v.half()
    _, v8, _, vs = tm.tilemix_quantize_qk(whole, v, v)
    best = []
    for height in (0.0, climb):
        k[:, :, 128:, 0] = height * d ** 0.5 / (8.0 * 1.4426950408889634)
        k16 = k.half()
        q8, _, qs, _ = tm.tilemix_quantize_qk(p, q, k16[:, :, ctx - L:])
        _, k8, _, ks = tm.tilemix_quantize_qk(whole, k16, k16)
        times = []
        for _ in range(8):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(4):
                tm.tilemix_attention_fwd_chunk_v8(p, ctx, q, k16, v8, vs, q8, k8, qs, ks, words)
            t1.record()
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1))
        best.append(min(times))
    assert best[1] < 1.4 * best[0], best
