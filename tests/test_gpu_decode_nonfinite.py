"""Decode over scores that are not finite: a row is finite, zero or NaN by what its keys, values and query hold, not by the number
of its splits, and its LSE agrees.  Part of a row without a single finite score has no weight beside the others."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
INF = float("inf")


def _run(R, L, lens, splits, change, d=128, tile=128):
    from paper_2608_17336_b200 import binding as tm
    B, Hk = len(lens), 2
    gen = torch.Generator().manual_seed(L + R)
    q = torch.randn((B, Hk * R, d), generator=gen).half()
    k, v = (torch.randn((B, Hk, L, d), generator=gen).half() for _ in range(2))
    q[..., 0] = 1.0                       # the channel that carries what is not finite
    change(q, k, v)
    q, k, v = q.to(DEV), k.to(DEV), v.to(DEV)
    k8, v8, ks, vs = tm.tilemix_quantize_qk(tm.problem(B, Hk, Hk, L, d, tile, tile), k, v)
    p = tm.decode_problem(B, Hk * R, Hk, d, L, tile, 1, n_splits=splits)
    r = tm.tilemix_decode_int8kv(p, q, k, k8, ks, v8, vs, None, torch.tensor(lens, dtype=torch.int32, device=DEV), want_lse=True)
    assert tm.tilemix_read_status(r["workspace"])[0] == 0
    return r["out"], r["lse"], q, k, v8, vs


def _no_score(q, k, v):
    k[..., 0] = -INF


def _no_score_in_256_keys(q, k, v):
    k[:, :, :256, 0] = -INF


def _nan_query(q, k, v):
    q[..., 5] = float("nan")


def _nan_key(q, k, v):
    k[:, :, 70, 0] = float("nan")


def _inf_key(q, k, v):
    k[:, :, 70, 0] = INF


def _inf_value(q, k, v):
    v[:, :, 70, 3] = INF


@pytest.mark.parametrize("R", [1, 2, 4, 8])
@pytest.mark.parametrize("splits", [1, 2, 3, -1])
def test_part_of_a_row_without_a_score(R, splits):
    """Of up to 512 keys the first 256 (with one split: all that one of the two softmax streams sees) score -inf."""
    lens = [512, 300, 200]
    out, lse, q, k, v8, vs = _run(R, 512, lens, splits, _no_score_in_256_keys)
    for b, n in enumerate(lens):
        if n <= 256:
            assert (out[b] == 0).all() and torch.isneginf(lse[b]).all()
            continue
        kd = k[b, :, 256:n].double().repeat_interleave(R, 0)
        vd = (v8[b].double() * vs[b].double().repeat_interleave(128, -1)[:, :, None])[:, 256:n].repeat_interleave(R, 0)
        s = torch.einsum("hd,hnd->hn", q[b].double(), kd) / 128 ** 0.5
        ref = torch.einsum("hn,hnd->hd", torch.softmax(s, -1), vd)
        # a probability is rounded to FP16 once (2^-11 of it), the output too
        assert (out[b].double() - ref).abs().max() < 2.0 ** -10 * vd.abs().max()
        assert (lse[b].double() - torch.logsumexp(s, -1)).abs().max() < 1e-4


@pytest.mark.parametrize("R", [1, 4, 8])
@pytest.mark.parametrize("d,tile", [(128, 128), (64, 64)])
@pytest.mark.parametrize("change,kind", [(_no_score, "zero"), (_nan_query, "zero"), (_nan_key, "zero"), (_inf_key, "zero"), (_inf_value, "nan")])
def test_kind_of_a_row_does_not_depend_on_the_splits(change, kind, d, tile, R):
    for lens in ([1000, 500], [200, 90]):
        for splits in (1, 2, 3, 0, -1):
            out, lse, *_ = _run(R, 1000, lens, splits, change, d, tile)
            if kind == "zero":
                assert (out == 0).all() and torch.isneginf(lse).all(), (lens, splits)
            else:
                assert torch.isnan(out).all() and torch.isfinite(lse).all(), (lens, splits)
