"""The quantiser's codes come from one fused multiply-add with a per-block factor; the definition is an IEEE quotient and a
round to even.  Blocks whose maximum runs over every binary16 mantissa (and the smallest magnitudes), filled with the values that could tell
the two apart: the binary16 neighbours of every half-integer multiple of delta, half of the maximum, the maximum."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [0, 1, 2, 8, 14, 15, 22, 29, 30])
def test_codes_next_to_half_integers_for_every_maximum(exponent):
    from paper_2608_17336_b200 import binding as tm
    d, blk = 64, 64
    bits = (exponent << 10) + np.arange(1024, dtype=np.int64)
    if exponent == 0:
        bits = np.maximum(bits, 1)
    amax = bits.astype(np.uint16).view(np.float16).astype(np.float64)
    near = ((np.arange(127) + 0.5)[None, :] * (amax / 127.0)[:, None]).astype(np.float16)
    b = near.view(np.uint16).astype(np.int64)
    cand = np.concatenate([np.clip(b + o, 0, bits[:, None]) for o in (-1, 0, 1)]
                          + [(amax / 2).astype(np.float16).view(np.uint16).astype(np.int64)[:, None], bits[:, None]], axis=1)
    x = np.zeros((1024, blk * d), np.uint16)
    x[:, :cand.shape[1]] = cand
    x[:, 1024:1024 + cand.shape[1]] = cand | 0x8000
    x = np.ascontiguousarray(x.reshape(1, 1, 1024 * blk, d))
    q8, qs = oracle.quantize(x, blk)
    t = torch.from_numpy(x.view(np.int16)).view(torch.float16).cuda()
    p = tm.problem(1, 1, 1, 1024 * blk, d, blk, blk, 1)
    strided = torch.zeros((1, 1, 1024 * blk, 2 * d), dtype=torch.float16, device="cuda")[..., :d]
    strided.copy_(t)
    for src in (t, strided):        # contiguous rows (streamed) and strided ones
        got = tm.tilemix_quantize_qk(p, src, src)
        for codes, scale in ((got[0], got[2]), (got[1], got[3])):
            assert np.array_equal(codes.cpu().numpy(), q8)
            assert np.array_equal(scale.cpu().numpy().view(np.uint32), qs.view(np.uint32))
