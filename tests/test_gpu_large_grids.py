"""Grids of more than half a wave, where a CTA has two tiles -- two adjacent ones of a head (odd head ratios) or the same
rows of two heads (even ones) -- for the forms whose other tests have small grids: a chunk against an INT8 value cache and
packed batches of several sequences, both head dimensions, whole and half-tile K blocks.  Some heads against the oracle;
every KV head bit for bit against a call on that head alone, which runs one tile per CTA."""
import numpy as np
import pytest
import torch

import oracle
from oracle import decode as od
from tests import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
HALF_WAVE = 74


def _keys(shape, axis, d, gen):
    """Neighbouring half tiles of clearly different scales: a step that takes another one's is far out of tolerance."""
    L = shape[axis]
    ramp = 1.0 + 2.0 * ((torch.arange(L) // (d // 2)) % 3)
    return (torch.randn(shape, generator=gen) * ramp.view([-1 if a == axis else 1 for a in range(len(shape))])).half()


def _close(got, ref, lse, ref_lse):
    got = got.float().cpu().numpy().astype(np.float64)
    err = np.abs(got - ref)
    assert (err <= H.ATOL * np.maximum(1.0, np.abs(ref))).all(), f"max err {err.max():.3e}"
    assert np.abs(lse.cpu().numpy().astype(np.float64) - ref_lse).max() < 2e-3


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("d,B,Hq,Hk,Lk,Lq", [(128, 2, 24, 12, 900, 388), (128, 1, 60, 20, 640, 384), (128, 1, 80, 20, 513, 129),
                                             (64, 2, 24, 12, 640, 512), (64, 1, 75, 25, 449, 321), (64, 2, 48, 12, 330, 138)])
def test_chunk_against_an_int8_value_cache(d, B, Hq, Hk, Lk, Lq, half):
    from paper_2608_17336_b200 import binding as tm
    blk_k = d // 2 if half else d
    rep, off = Hq // Hk, Lk - Lq
    assert off % d == 0 and B * Hq * -(-Lq // (2 * 128)) > HALF_WAVE
    gen = torch.Generator().manual_seed(Lk + d)
    q, v = torch.randn((B, Hq, Lq, d), generator=gen).half(), (torch.randn((B, Hk, Lk, d), generator=gen) * 1.5).half()
    k = _keys((B, Hk, Lk, d), 2, d, gen)
    po = oracle.Problem(B, Hk, Hk, Lk, d, d, d, 2)
    route = (np.random.default_rng(Lq).random((1, Hk, po.T_m, po.T_mask)) < 0.5).astype(np.uint8)
    q8, qs = oracle.quantize(H.np_bits(q), d)
    k8, ks = oracle.quantize(H.np_bits(k), blk_k)
    v8, vs = oracle.quantize(H.np_bits(v), d)
    words, _ = oracle.pack(po, route)
    dev = lambda a: torch.from_numpy(a).to(DEV)  # noqa: E731
    wd = dev(words.view(np.int32))

    def run(b, hq, hk):          # slices of sequences, query heads, KV heads
        t = [dev(np.ascontiguousarray(x[b, s])) for x, s in ((v8, hk), (vs, hk), (q8, hq), (k8, hk), (qs, hq), (ks, hk))]
        p = tm.problem(b.stop - b.start, hq.stop - hq.start, hk.stop - hk.start, Lq, d, d, d, 2, quant_blk_k=blk_k)
        r = tm.tilemix_attention_fwd_chunk_v8(p, Lk, q[b, hq].contiguous().to(DEV), k[b, hk].contiguous().to(DEV), *t,
                                              wd[:, hk].contiguous(), want_lse=True)
        assert tm.tilemix_read_status(r["workspace"])[0] == 0
        return r["out"], r["lse"]
    out, lse = run(slice(0, B), slice(0, Hq), slice(0, Hk))
    for h in sorted({0, rep - 1, Hq - 1}):
        g = h // rep
        ref, ref_lse = od.chunk_v8(H.np_bits(q[:, h:h + 1]), q8[:, h:h + 1], qs[:, h:h + 1], H.np_bits(k[:, g:g + 1]), k8[:, g:g + 1],
                                   ks[:, g:g + 1], v8[:, g:g + 1], vs[:, g:g + 1], words[:, g:g + 1], d, 2, blk_k=blk_k)
        _close(out[:, h:h + 1], ref, lse[:, h:h + 1], ref_lse)
    for b in range(B):
        for g in range(Hk):
            hs = slice(g * rep, (g + 1) * rep)
            o1, l1 = run(slice(b, b + 1), hs, slice(g, g + 1))
            assert torch.equal(o1[0], out[b, hs]) and torch.equal(l1[0], lse[b, hs]), (b, g)


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("d,Hq,Hk,lens", [(128, 16, 8, [300, 0, 129, 641, 5, 128, 1000]), (128, 21, 7, [385, 70, 0, 900, 257]),
                                          (128, 32, 8, [1, 500, 130, 260]), (64, 24, 12, [200, 1, 0, 449, 65, 128, 330]),
                                          (64, 33, 11, [321, 64, 193, 500, 0, 90]), (64, 40, 10, [129, 130, 400])])
def test_packed_batch_of_several_sequences(d, Hq, Hk, lens, half):
    from paper_2608_17336_b200 import binding as tm
    blk_k, rep, G = (d // 2 if half else d), Hq // Hk, 2
    cu = np.cumsum([0] + lens).tolist()
    assert Hq * sum(-(-n // 256) for n in lens) > HALF_WAVE
    gen = torch.Generator().manual_seed(sum(lens) + Hq)
    q, v = torch.randn((cu[-1], Hq, d), generator=gen).half(), torch.randn((cu[-1], Hk, d), generator=gen).half()
    k = _keys((cu[-1], Hk, d), 0, d, gen)
    vl = tm.Varlen(cu)
    n = tm.tilemix_varlen_counts(tm.problem(1, Hq, Hk, cu[-1], d, d, d, G, quant_blk_k=blk_k), vl)
    route = (np.random.default_rng(Hq).random((Hk, n["sum_T_m"], n["T_mask_max"])) < 0.5).astype(np.uint8)

    def run(hq, hk):
        p = tm.problem(1, hq.stop - hq.start, hk.stop - hk.start, cu[-1], d, d, d, G, quant_blk_k=blk_k)
        qd, kd, vd = (x[:, s].contiguous().to(DEV) for x, s in ((q, hq), (k, hk), (v, hk)))
        codes = tm.tilemix_quantize_qk_varlen(p, vl, qd, kd)
        words, _ = tm.tilemix_pack_routing_mask_varlen(p, vl, torch.from_numpy(route[hk].copy()).to(DEV))
        r = tm.tilemix_attention_fwd_varlen(p, vl, qd, kd, vd, *codes, words, want_lse=True)
        assert tm.tilemix_read_status(r["workspace"])[0] == 0
        return r["out"], r["lse"]
    out, lse = run(slice(0, Hq), slice(0, Hk))
    row0 = 0
    for s, length in enumerate(lens):
        t_m = -(-length // d)
        if length:
            po = oracle.Problem(1, rep, 1, length, d, d, d, G, blk_q=d, blk_k=blk_k)
            at = slice(cu[s], cu[s + 1])
            for g in {0, Hk - 1}:
                hs = slice(g * rep, (g + 1) * rep)
                qb, kb, vb = (H.np_bits(x[at, h].permute(1, 0, 2)[None]) for x, h in ((q, hs), (k, slice(g, g + 1)), (v, slice(g, g + 1))))
                q8, qs = oracle.quantize(qb, d)
                k8, ks = oracle.quantize(kb, blk_k)
                words, _ = oracle.pack(po, np.ascontiguousarray(route[None, g:g + 1, row0:row0 + t_m, :po.T_mask]))
                ref, ref_lse, _ = oracle.attention_full(po, qb, kb, vb, q8, k8, qs, ks, words)
                _close(out[at, hs], ref[0].transpose(1, 0, 2), lse[hs, at], ref_lse[0])
        row0 += t_m
    for g in range(Hk):
        hs = slice(g * rep, (g + 1) * rep)
        o1, l1 = run(hs, slice(g, g + 1))
        assert torch.equal(o1, out[:, hs]) and torch.equal(l1, lse[hs]), g
