"""Grouped queries: a CTA whose two tiles are the same rows of two query heads of one KV head (grids of more than half a
wave, an even number of query heads per KV head).  Rows and debug tiles against the oracle at odd numbers of tiles, an odd
head ratio beside it, and bit-identity of the operand modes, of a packed one-sequence batch and of a chunk."""
import numpy as np
import pytest
import torch

import oracle
from tests import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("B,Hq,Hk,L,d,G,blk_k", [(2, 32, 8, 700, 128, 1, 128), (1, 48, 24, 900, 128, 2, 64), (1, 60, 20, 650, 128, 1, 128),
                                                 (2, 32, 4, 700, 64, 1, 64), (3, 80, 40, 130, 64, 1, 32)])
def test_rows_modes_packed_and_chunk(B, Hq, Hk, L, d, G, blk_k):
    from paper_2608_17336_b200 import binding as tm
    gen = torch.Generator().manual_seed(L + Hq)
    q = torch.randn((B, Hq, L, d), generator=gen).half()
    k = (torch.randn((B, Hk, L, d), generator=gen) * (1.0 + 2.0 * ((torch.arange(L) // d) % 2)).view(1, 1, L, 1)).half()
    v = torch.randn((B, Hk, L, d), generator=gen).half()
    po = oracle.Problem(B, Hq, Hk, L, d, d, d, G, blk_q=d, blk_k=blk_k)
    route = (np.random.default_rng(L).random((1, Hk, po.T_m, po.T_mask)) < 0.5).astype(np.uint8)
    qb, kb, vb = H.np_bits(q), H.np_bits(k), H.np_bits(v)
    q8, qs = oracle.quantize(qb, d)
    k8, ks = oracle.quantize(kb, blk_k)
    wo, _ = oracle.pack(po, route, False)
    rows = [(b, h, i) for b in range(B) for h in range(Hq) for i in sorted({0, L - 1, d - 1, d, L // 2, 2 * d % L, (h * 37) % L})]
    ref, ref_lse, _ = oracle.attention_rows(po, qb, kb, vb, q8, k8, qs, ks, wo, rows)

    p = tm.problem(B, Hq, Hk, L, d, d, d, G, quant_blk_k=blk_k)
    qd, kd, vd = q.to(DEV), k.to(DEV), v.to(DEV)
    codes = tm.tilemix_quantize_qk(p, qd, kd)
    words, _ = tm.tilemix_pack_routing_mask(p, torch.from_numpy(route).to(DEV))
    res = tm.tilemix_attention_fwd(p, qd, kd, vd, *codes, words, want_lse=True)
    assert tm.tilemix_read_status(res["workspace"])[0] == 0
    H.check_rows(res["out"], ref, rows)
    lse = np.array([res["lse"][r].item() for r in rows])
    assert np.abs(lse - ref_lse).max() < 2e-3
    tiles = [(B - 1, h, m, n) for h in (0, 1, Hq - 1) for m in range(po.T_m) for n in range(m + 1)]
    dbg = tm.tilemix_attention_fwd(p, qd, kd, vd, *codes, words, debug_tiles=tiles)
    raw, kind = dbg["raw"].cpu().numpy(), dbg["kind"].cpu().numpy()
    for e, t in enumerate(tiles):
        assert kind[e] == route[0, t[1] // (Hq // Hk), t[2], t[3] // G]
        if kind[e]:
            assert np.array_equal(raw[e], oracle.int32_tile(po, q8, k8, *t)), t
    if d == 128 and blk_k == d:
        otf = tm.tilemix_attention_fwd(tm.problem(B, Hq, Hk, L, d, d, d, G, flags=tm.QUANT_ON_THE_FLY), qd, kd, vd, words=words, want_lse=True)
        assert torch.equal(otf["out"], res["out"]) and torch.equal(otf["lse"], res["lse"])
    # the first sequence as a packed batch of one, and its last rows as a chunk
    one = tm.problem(1, Hq, Hk, L, d, d, d, G, quant_blk_k=blk_k)
    vl = tm.Varlen([0, L])
    tok = lambda x: x[0].transpose(0, 1).contiguous()  # noqa: E731
    cv = tm.tilemix_quantize_qk_varlen(one, vl, tok(qd), tok(kd))
    rv = tm.tilemix_attention_fwd_varlen(one, vl, tok(qd), tok(kd), tok(vd), *cv, words[0], want_lse=True)
    assert torch.equal(rv["out"], tok(res["out"])) and torch.equal(rv["lse"], res["lse"][0])
    off = d * (po.T_m // 2)
    if off:
        pc = tm.problem(B, Hq, Hk, L - off, d, d, d, G, quant_blk_k=blk_k)
        rc = tm.tilemix_attention_fwd_chunk(pc, L, qd[:, :, off:].contiguous(), kd, vd, codes[0][:, :, off:].contiguous(), codes[1],
                                            codes[2][:, :, off // d:].contiguous(), codes[3], words, want_lse=True)
        assert torch.equal(rc["out"], res["out"][:, :, off:]) and torch.equal(rc["lse"], res["lse"][:, :, off:])
