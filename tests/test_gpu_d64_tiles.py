"""Head dimension 64: the fused kernel's 128 x 128 accumulators carry 2 x 2 routing tiles.  Every row against the oracle
at the lengths where a tile's second row or key half is partial or missing, for both widths of the K quantisation
blocks, and chunks that begin in the middle of a 128-key tile.  The small batches run one tile per CTA, the large ones
two."""
import numpy as np
import pytest
import torch

import oracle
from tests import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _case(B, Hq, Hk, L, G, blk_k, f8, seed):
    from paper_2608_17336_b200 import binding as tm
    gen = torch.Generator().manual_seed(seed)
    # key blocks of clearly different scales: a step that takes the wrong one is far out of tolerance
    k = torch.randn((B, Hk, L, 64), generator=gen) * (1.0 + 2.0 * ((torch.arange(L) // 32) % 3)).view(1, 1, L, 1)
    q, v = torch.randn((B, Hq, L, 64), generator=gen).half(), torch.randn((B, Hk, L, 64), generator=gen).half()
    k = k.half()
    po = oracle.Problem(B, Hq, Hk, L, 64, 64, 64, G, blk_q=64, blk_k=blk_k)
    route = (np.random.default_rng(seed).random((1, Hk, po.T_m, po.T_mask)) < f8).astype(np.uint8)
    qb, kb, vb = H.np_bits(q), H.np_bits(k), H.np_bits(v)
    q8, qs = oracle.quantize(qb, 64)
    k8, ks = oracle.quantize(kb, blk_k)
    words, _ = oracle.pack(po, route, False)
    ref, ref_lse, _ = oracle.attention_full(po, qb, kb, vb, q8, k8, qs, ks, words)
    p = tm.problem(B, Hq, Hk, L, 64, 64, 64, G, quant_blk_k=blk_k)
    qd, kd, vd = q.to(DEV), k.to(DEV), v.to(DEV)
    codes = tm.tilemix_quantize_qk(p, qd, kd)
    wd, _ = tm.tilemix_pack_routing_mask(p, torch.from_numpy(route).to(DEV))
    return tm, p, po, (qd, kd, vd), codes, wd, (q8, k8), ref, ref_lse


def _close(res, ref, ref_lse):
    got = res["out"].float().cpu().numpy().astype(np.float64)
    assert (np.abs(got - ref) <= H.ATOL * np.maximum(1.0, np.abs(ref))).all(), np.abs(got - ref).max()
    assert np.abs(res["lse"].cpu().numpy() - ref_lse).max() < 2e-3


@pytest.mark.parametrize("blk_k", [64, 32])
@pytest.mark.parametrize("B,Hq,Hk,L,G", [(1, 1, 1, 1, 1), (1, 2, 1, 64, 1), (1, 2, 2, 65, 1), (1, 2, 1, 128, 1), (1, 2, 2, 129, 1),
                                         (2, 2, 1, 200, 2), (1, 2, 1, 321, 1), (1, 1, 1, 449, 3), (2, 40, 40, 257, 1),
                                         (1, 80, 20, 100, 1)])
def test_all_rows_at_tile_edges(B, Hq, Hk, L, G, blk_k):
    tm, p, po, (q, k, v), codes, words, (q8, k8), ref, ref_lse = _case(B, Hq, Hk, L, G, blk_k, 0.5, seed=L + blk_k)
    res = tm.tilemix_attention_fwd(p, q, k, v, *codes, words, want_lse=True)
    assert tm.tilemix_read_status(res["workspace"])[0] == 0
    _close(res, ref, ref_lse)
    tiles = [(b, h, m, n) for b in range(B) for h in range(min(Hq, 3)) for m in range(po.T_m) for n in range(m + 1)]
    dbg = tm.tilemix_attention_fwd(p, q, k, v, *codes, words, want_lse=True, debug_tiles=tiles)
    _close(dbg, ref, ref_lse)
    raw, kind = dbg["raw"].cpu().numpy(), dbg["kind"].cpu().numpy()
    for e, (b, h, m, n) in enumerate(tiles):
        assert kind[e] in (0, 1)
        if kind[e]:
            assert np.array_equal(raw[e], oracle.int32_tile(po, q8, k8, b, h, m, n)), tiles[e]


@pytest.mark.parametrize("blk_k", [64, 32])
@pytest.mark.parametrize("L,off", [(200, 64), (330, 192), (512, 320), (449, 256), (129, 64)])
def test_chunk_beginning_inside_a_key_tile(L, off, blk_k):
    tm, p, po, (q, k, v), codes, words, _, ref, ref_lse = _case(1, 2, 1, L, 1, blk_k, 0.5, seed=L)
    full = tm.tilemix_attention_fwd(p, q, k, v, *codes, words, want_lse=True)
    _close(full, ref, ref_lse)
    pc = tm.problem(1, 2, 1, L - off, 64, 64, 64, 1, quant_blk_k=blk_k)
    q8c, qsc = codes[0][:, :, off:].contiguous(), codes[2][:, :, off // 64:].contiguous()
    res = tm.tilemix_attention_fwd_chunk(pc, L, q[:, :, off:].contiguous(), k, v, q8c, codes[1], qsc, codes[3], words, want_lse=True)
    assert tm.tilemix_read_status(res["workspace"])[0] == 0
    assert torch.equal(res["out"].view(torch.int16), full["out"][:, :, off:].contiguous().view(torch.int16))
    assert torch.equal(res["lse"], full["lse"][:, :, off:])
