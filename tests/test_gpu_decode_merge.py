"""A row with one CTA, and the merge of splits inside the step (the CTAs of a row count their arrivals), on both sides of the line to the
merge kernel: few and many splits, a last split of one tile, empty sequences, an odd number of rows (two rows share a counter
word), repeated calls on one workspace whose counters hold garbage before each."""
import numpy as np
import pytest
import torch

from oracle import decode as od

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("B,Hq,Hk,d,tile,L,splits", [(1, 8, 1, 128, 128, 3000, 0), (3, 12, 3, 128, 128, 1100, 9), (3, 6, 3, 128, 128, 1500, -1),
                                                     (1, 4, 4, 64, 64, 4000, 0), (5, 10, 5, 64, 128, 700, 3), (3, 24, 3, 128, 64, 1000, 5),
                                                     (5, 20, 5, 128, 128, 900, 1), (5, 40, 5, 128, 128, 700, 1), (5, 10, 5, 64, 128, 700, 1), (5, 10, 5, 128, 64, 400, 1), (5, 8, 2, 128, 128, 2000, -1),
                                                     (2, 148, 37, 128, 128, 300, 2), (2, 148, 74, 128, 128, 300, 2), (2, 75, 75, 64, 64, 500, 2)])
def test_merge_in_the_step_against_the_oracle(B, Hq, Hk, d, tile, L, splits):
    from paper_2608_17336_b200 import binding as tm
    gen = torch.Generator().manual_seed(L + Hq)
    q = torch.randn((B, Hq, d), generator=gen).half()
    k, v = (torch.randn((B, Hk, L, d), generator=gen).half() for _ in range(2))
    lens = [L, 0, tile + 1, L - 1, 1][:B]
    route = (np.random.default_rng(L).random((1, Hk, -(-L // tile))) < 0.5).astype(np.uint8)
    k8, v8, ks, vs = tm.tilemix_quantize_qk(tm.problem(B, Hk, Hk, L, d, tile, tile), k.to(DEV), v.to(DEV))
    words = torch.from_numpy(od.pack_row(route).view(np.int32)).to(DEV)
    p = tm.decode_problem(B, Hq, Hk, d, L, tile, 1, n_splits=splits)
    ws = torch.empty(tm.tilemix_decode_workspace_size(p), dtype=torch.uint8, device=DEV)
    outs = []
    for fill in (0xff, 0x5a, 0x01):
        ws.fill_(fill)
        r = tm.tilemix_decode_int8kv(p, q.to(DEV), k.to(DEV), k8, ks, v8, vs, words, torch.tensor(lens, dtype=torch.int32, device=DEV),
                                     want_lse=True, workspace=ws)
        assert tm.tilemix_read_status(ws)[0] == 0
        outs.append((r["out"].clone(), r["lse"].clone()))
    for o in outs[1:]:
        assert torch.equal(o[0], outs[0][0]) and torch.equal(o[1], outs[0][1])
    # the definition in float64 over the same codes: probabilities are rounded to FP16 (2^-11 each), sums are FP32
    rep = Hq // Hk
    dec = lambda x, s: x.double().cpu() * s.double().cpu().repeat_interleave(tile, -1)[..., :L, None]  # noqa: E731
    kd, vd = dec(k8, ks), dec(v8, vs)
    amax = q.abs().amax(-1, keepdim=True).float()
    dq = amax / 127.0
    q8 = torch.round(q.float() / dq).double() * dq.double()
    for b in range(B):
        n = lens[b]
        if n == 0:
            assert (outs[0][0][b] == 0).all() and torch.isneginf(outs[0][1][b]).all()
            continue
        for h in range(Hq):
            g = h // rep
            int8 = torch.from_numpy(route[0, g].repeat(tile)[:n].astype(bool))
            s = torch.where(int8, kd[b, g, :n] @ q8[b, h], k[b, g, :n].double() @ q[b, h].double()) / d ** 0.5
            ref = torch.softmax(s, 0) @ vd[b, g, :n]
            assert (outs[0][0][b, h].double().cpu() - ref).abs().max() < 2e-3 * max(1.0, ref.abs().max().item()), (b, h)
            assert abs(outs[0][1][b, h].item() - torch.logsumexp(s, 0).item()) < 2e-3


def _decode(tm, q, k, v, lens, tile, splits):
    B, Hk, L, d = k.shape
    k8, v8, ks, vs = tm.tilemix_quantize_qk(tm.problem(B, Hk, Hk, L, d, tile, tile), k, v)
    words = torch.full((1, Hk, -(-(-(-L // tile)) // 32)), 0x33333333, dtype=torch.int32, device=DEV)
    p = tm.decode_problem(B, q.shape[1], Hk, d, L, tile, 1, n_splits=splits)
    ws = torch.empty(tm.tilemix_decode_workspace_size(p), dtype=torch.uint8, device=DEV)
    before = tm.tilemix_launch_count()
    r = tm.tilemix_decode_int8kv(p, q, k, k8, ks, v8, vs, words, torch.tensor(lens, dtype=torch.int32, device=DEV), want_lse=True,
                                 workspace=ws)
    launches = tm.tilemix_launch_count() - before
    assert tm.tilemix_read_status(ws)[0] == 0
    return r["out"], r["lse"], launches


# (B, Hk, R, d, tile, L, splits): launches of the call
ROUTES = [((2, 2, 4, 128, 128, 3000, 1), 2), ((2, 2, 4, 128, 128, 3000, 2), 3), ((2, 2, 4, 128, 128, 3000, 3), 2),
          ((25, 2, 4, 128, 128, 600, 3), 3),                # 150 CTAs: more than a wave
          ((3, 2, 4, 128, 128, 3000, -1), 2), ((60, 2, 1, 128, 128, 700, -1), 2), ((80, 2, 1, 128, 128, 300, -1), 2),
          ((2, 2, 4, 128, 64, 600, 1), 2), ((2, 2, 4, 128, 64, 600, 2), 3), ((2, 2, 4, 128, 64, 450, 4), 3),   # two tiles a split
          ((2, 2, 4, 128, 64, 600, 4), 2), ((2, 2, 4, 128, 64, 320, 5), 2),
          ((2, 2, 8, 64, 64, 1000, 4), 3), ((2, 2, 8, 64, 128, 1100, 4), 2), ((50, 2, 1, 64, 64, 1200, 3), 3)]  # 300 CTAs


@pytest.mark.parametrize("case,launches", ROUTES)
def test_kernels_of_a_step(case, launches):
    """Where the step merges, or has nothing to merge, there are two kernels; with the merge kernel three."""
    from paper_2608_17336_b200 import binding as tm
    B, Hk, R, d, tile, L, splits = case
    gen = torch.Generator(device=DEV).manual_seed(1)
    q, k, v = (torch.randn(s, generator=gen, device=DEV).half() for s in ((B, Hk * R, d), (B, Hk, L, d), (B, Hk, L, d)))
    assert _decode(tm, q, k, v, [L] * B, tile, splits)[2] == launches


@pytest.mark.parametrize("R", [1, 2, 4, 8])
@pytest.mark.parametrize("d,tile,splits", [(128, 128, 3), (128, 128, 4), (128, 128, 5), (128, 128, 17), (128, 64, 5), (128, 64, 8), (128, 64, 33),
                                           (64, 64, 7), (64, 128, 16)])
def test_same_bits_from_the_step_and_the_merge_kernel(d, tile, splits, R):
    """The first sequences alone are merged in the step; in a batch of several waves, by the kernel."""
    from paper_2608_17336_b200 import binding as tm
    Hk, L = 3, 128 * splits
    B = -(-300 // (Hk * splits)) + 1
    gen = torch.Generator(device=DEV).manual_seed(splits + R)
    q, k, v = (torch.randn(s, generator=gen, device=DEV).half() for s in ((B, Hk * R, d), (B, Hk, L, d), (B, Hk, L, d)))
    lens = [L, L - 77] + [L] * (B - 2)
    many = _decode(tm, q, k, v, lens, tile, splits)
    few = _decode(tm, q[:2].contiguous(), k[:2].contiguous(), v[:2].contiguous(), lens[:2], tile, splits)
    assert (few[2], many[2]) == (2, 3)
    assert torch.equal(few[0], many[0][:2]) and torch.equal(few[1], many[1][:2])
