"""Head dimension 64: a tile of the fused kernel is 2 x 2 routing tiles, so the first 64 rows of one take part in a step
whose keys all lie above their diagonal.  A key or value that is not finite there must not reach them: every row before
the routing tile that holds it keeps its bits, in each form of the kernel."""
import pytest
import torch

pytestmark = pytest.mark.gpu
T = 64


def _inputs(B, Hq, Hk, L, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn((B, h, L, T), generator=gen, device="cuda").half() for h in (Hq, Hk, Hk)]


def _route(p, f8, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.rand((1, p.heads_kv, p.T_m, p.T_mask), generator=gen, device="cuda") < f8).to(torch.uint8)


def _dense(q, k, v, blk_k, f8):
    from paper_2608_17336_b200 import binding as tm
    p = tm.problem(q.shape[0], q.shape[1], k.shape[1], q.shape[2], T, T, T, 1, quant_blk_k=blk_k)
    codes = tm.tilemix_quantize_qk(p, q, k)
    words, _ = tm.tilemix_pack_routing_mask(p, _route(p, f8, 5))
    r = tm.tilemix_attention_fwd(p, q, k, v, *codes, words, want_lse=True)
    assert tm.tilemix_read_status(r["workspace"])[0] == 0
    return r["out"], r["lse"]


@pytest.mark.parametrize("blk_k", [64, 32])
@pytest.mark.parametrize("f8", [0.0, 0.5, 1.0])
@pytest.mark.parametrize("B,Hq,Hk", [(1, 2, 1), (2, 40, 40), (2, 40, 20)])     # one tile per CTA, two adjacent ones, head pairs
def test_rows_before_the_tile_keep_their_bits(B, Hq, Hk, f8, blk_k):
    L = 449
    q, k, v = _inputs(B, Hq, Hk, L, 3)
    out, lse = _dense(q, k, v, blk_k, f8)
    assert torch.isfinite(out).all() and torch.isfinite(lse).all()
    for tile in (1, 2, 3, 6):
        for at, bad in ((tile * T, float("nan")), (min(L, (tile + 1) * T) - 1, float("inf"))):
            k2, v2 = k.clone(), v.clone()
            k2[:, :, at, 9] = bad
            v2[:, :, at, 11] = -bad
            o2, l2 = _dense(q, k2, v2, blk_k, f8)
            assert torch.equal(o2[:, :, :tile * T], out[:, :, :tile * T]), (tile, bad)
            assert torch.equal(l2[:, :, :tile * T], lse[:, :, :tile * T]), (tile, bad)
            assert not torch.isfinite(o2[:, :, at:, 11]).any()


@pytest.mark.parametrize("Hq,Hk", [(2, 1), (40, 40), (80, 40)])
def test_next_sequence_of_a_packed_batch(Hq, Hk):
    """The first tokens of the next sequence lie in the last key tile of this one; the rows of its earlier routing tiles
    do not see them."""
    from paper_2608_17336_b200 import binding as tm
    cu = [0, 2 * T + T // 2 + T, 2 * T + T // 2 + T + 300]
    n0 = cu[1]
    p, vl = tm.problem(1, Hq, Hk, cu[-1], T, T, T, 1), tm.Varlen(cu)
    n = tm.tilemix_varlen_counts(p, vl)
    gen = torch.Generator(device="cuda").manual_seed(4)
    q, k, v = (torch.randn((cu[-1], h, T), generator=gen, device="cuda").half() for h in (Hq, Hk, Hk))
    route = (torch.rand((Hk, n["sum_T_m"], n["T_mask_max"]), generator=gen, device="cuda") < 0.5).to(torch.uint8)

    def run(k, v):
        codes = tm.tilemix_quantize_qk_varlen(p, vl, q, k)
        words, _ = tm.tilemix_pack_routing_mask_varlen(p, vl, route)
        return tm.tilemix_attention_fwd_varlen(p, vl, q, k, v, *codes, words)["out"]
    out = run(k, v)
    k2, v2 = k.clone(), v.clone()
    k2[n0:n0 + 40, :, 3] = float("nan")
    v2[n0:n0 + 40, :, 5] = float("inf")
    edge = n0 // T * T
    assert torch.equal(run(k2, v2)[:edge], out[:edge])


@pytest.mark.parametrize("Hq,Hk,off", [(2, 1, T), (2, 1, 2 * T), (40, 40, T), (80, 40, 3 * T)])
def test_chunk_and_int8_value_cache(Hq, Hk, off):
    from paper_2608_17336_b200 import binding as tm
    L = 449
    q, k, v = _inputs(1, Hq, Hk, L, 6)
    p = tm.problem(1, Hq, Hk, L, T, T, T, 1)
    pc = tm.problem(1, Hq, Hk, L - off, T, T, T, 1)
    words, _ = tm.tilemix_pack_routing_mask(p, _route(p, 0.5, 7))

    def run(k, v):
        q8, k8, qs, ks = tm.tilemix_quantize_qk(p, q, k)
        _, v8, _, vs = tm.tilemix_quantize_qk(tm.problem(1, Hk, Hk, L, T, T, T), k, v)
        a = (q[:, :, off:].contiguous(), k), (q8[:, :, off:].contiguous(), k8, qs[:, :, off // T:].contiguous(), ks, words)
        return (tm.tilemix_attention_fwd_chunk(pc, L, *a[0], v, *a[1])["out"],
                tm.tilemix_attention_fwd_chunk_v8(pc, L, *a[0], v8, vs, *a[1])["out"])
    want = run(k, v)
    for tile in range(off // T + 1, 7):
        k2, v2 = k.clone(), v.clone()
        k2[:, :, tile * T + 1, 0] = float("nan")
        v2[:, :, tile * T + 1, 2] = float("inf")
        for w, got in zip(want, run(k2, v2)):
            assert torch.equal(got[:, :, :tile * T - off], w[:, :, :tile * T - off]), tile
