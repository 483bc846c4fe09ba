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
