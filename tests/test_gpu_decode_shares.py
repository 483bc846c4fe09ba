"""Warp-level decode form: two 64-key routing tiles per kernel tile, and a grid that takes sequences of unequal length
longest first -- one to eight sequences per lane of the warp that orders them, lengths at the edges of kernel and routing
tiles, more sequences than are ordered; a sequence's result does not depend on the sequences beside it.  The tcgen05
form with CTAs shared out over the rows, two waves of them."""
import numpy as np
import pytest
import torch

from tests.test_gpu_decode import _case, _check, _gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,tile", [(64, 64), (64, 128), (128, 64)])
@pytest.mark.parametrize("B,Hq,Hk,L,G,splits", [(1, 2, 1, 700, 1, 0), (5, 4, 2, 1500, 3, 0), (33, 4, 4, 400, 1, -1), (100, 8, 1, 300, 2, 0),
                                                (200, 2, 2, 260, 1, 0), (4, 2, 1, 900, 1, 3), (4, 2, 1, 900, 1, 1000)])
def test_unequal_lengths(B, Hq, Hk, L, G, splits, d, tile):
    rng = np.random.default_rng(B + L)
    lens = rng.integers(0, L + 1, B)
    edges = [L, 0, 1, 64, 65, 127, 128, 129, 192, 193, 256]
    lens[:min(B, len(edges))] = [min(L, e) for e in edges[:B]]
    q, k, v, route, lens = _case(B, Hq, Hk, L, d, tile, G, seed=B, lens=lens)
    _check(q, k, v, route, lens, tile, G, n_splits=splits)


def test_more_sequences_than_are_ordered():
    q, k, v, route, lens = _case(300, 1, 1, 200, 64, 64, 1, seed=3, lens=np.arange(300) % 201)
    _check(q, k, v, route, lens, 64, 1)


@pytest.mark.parametrize("splits", [0, -1, 5])
@pytest.mark.parametrize("d,tile", [(64, 64), (64, 128), (128, 64), (128, 128)])
@pytest.mark.parametrize("B", [6, 40])
def test_a_sequence_does_not_depend_on_the_lengths_beside_it(B, d, tile, splits):
    """Same bits whatever the other sequences' lengths are, and in a repeated call; every length 0 included.  (In the
    tcgen05 form -1 shares CTAs out by the lengths.)"""
    if (d, tile, splits) == (128, 128, -1):
        splits = 1
    L = 1500
    first = np.random.default_rng(B).integers(1, L + 1, B)
    keep = np.arange(B) % 3 == 0
    runs = []
    for others in (first, first, np.full(B, L), np.zeros(B, np.int64), first[::-1]):
        lens = np.where(keep, first, others)
        q, k, v, route, lens = _case(B, 4, 2, L, d, tile, 2, seed=5, lens=lens)
        res, _ = _gpu(q, k, v, route, lens, tile, 2, n_splits=splits)
        runs.append((res["out"][keep].cpu(), res["lse"][keep].cpu()))
    for out, lse in runs[1:]:
        assert torch.equal(out, runs[0][0]) and torch.equal(lse, runs[0][1])
    q, k, v, route, lens = _case(B, 4, 2, L, d, tile, 2, seed=5, lens=np.zeros(B))
    _check(q, k, v, route, np.append(lens[:-1], 1).astype(np.int32), tile, 2, n_splits=splits)
    res, _ = _gpu(q, k, v, route, lens, tile, 2, n_splits=splits)
    assert not res["out"].any() and torch.isneginf(res["lse"]).all()


@pytest.mark.parametrize("B,Hq,Hk,L,G", [(10, 16, 8, 1000, 1), (40, 8, 4, 400, 2), (80, 2, 2, 300, 1)])
def test_kernel_chosen_splits_with_more_rows_than_half_a_wave(B, Hq, Hk, L, G):
    """head_dim 128 with 128-key routing tiles: two waves of CTAs are shared out."""
    lens = np.random.default_rng(B).integers(0, L + 1, B)
    lens[:6] = [L, 0, 1, 64, 129, 200]
    q, k, v, route, lens = _case(B, Hq, Hk, L, 128, 128, G, seed=B, lens=lens)
    _check(q, k, v, route, lens, 128, G, n_splits=-1)
    _check(q, k, v, np.ones_like(route), lens, 128, G, n_splits=-1, k16_none=True)
