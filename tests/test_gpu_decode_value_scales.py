"""Decode against a value cache whose block scales are near 480: a probability times its block's scale has to fit FP16 while
the running maximum lags behind the one key of a step that climbs."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("climb", [5.0, 7.2, 7.9, 8.5, 12.0])
@pytest.mark.parametrize("R", [1, 4, 8])
@pytest.mark.parametrize("d,tile,every", [(128, 128, 256), (128, 64, 64), (64, 64, 128)])
def test_one_key_a_step_climbs(d, tile, every, R, climb):
    """`every`: the keys of a step of one of the form's streams.  In the tcgen05 form steps alternate between two streams, so
    two steps in a row carry the same score."""
    from paper_2608_17336_b200 import binding as tm
    B, Hk, L = 1, 2, 10 * every + 40
    gen = torch.Generator(device=DEV).manual_seed(int(10 * climb) + R)
    q = 0.1 * torch.randn((B, Hk * R, d), generator=gen, device=DEV)
    k, v = (torch.randn((B, Hk, L, d), generator=gen, device=DEV) for _ in range(2))
    k = 0.1 * k
    q[..., 0] = 8.0
    k[..., 0] = 0.0
    at = torch.arange(0, L, every, device=DEV)
    k[:, :, at, 0] = (at // every // 2) * climb * d ** 0.5 / (8.0 * 1.4426950408889634)
    v = torch.sign(v) * 61000.0 * (0.5 + 0.5 * torch.rand(v.shape, generator=gen, device=DEV))
    q, k, v = q.half(), k.half(), v.half()
    k8, v8, ks, vs = tm.tilemix_quantize_qk(tm.problem(B, Hk, Hk, L, d, tile, tile), k, v)
    rows = lambda s: s.double().repeat_interleave(tile, -1)[..., :L, None]  # noqa: E731
    vd = (v8.double() * rows(vs))[0].repeat_interleave(R, 0)
    for words, kd in ((None, k[0].double()), (torch.full((1, Hk, -(-(-(-L // tile)) // 32)), -1, dtype=torch.int32, device=DEV), (k8.double() * rows(ks))[0])):
        qd = q[0].double()
        if words is not None:
            delta = q[0].float().abs().amax(-1, keepdim=True) / 127.0
            qd = torch.round(q[0].float() / delta).double() * delta.double()
        s = torch.einsum("hd,hnd->hn", qd, kd.repeat_interleave(R, 0)) / d ** 0.5
        ref = torch.einsum("hn,hnd->hd", torch.softmax(s, -1), vd)
        for splits in (1, 2, 3):
            p = tm.decode_problem(B, Hk * R, Hk, d, L, tile, 1, n_splits=splits)
            out = tm.tilemix_decode_int8kv(p, q, k, k8, ks, v8, vs, words, torch.tensor([L], dtype=torch.int32, device=DEV))["out"][0]
            assert torch.isfinite(out).all()
            # a scaled probability and an output are rounded to FP16 once each (2^-11 of at most the largest value)
            assert (out.double() - ref).abs().max() < (2.0 ** -10 + 2.0 ** -14) * vd.abs().max(), splits
