"""The arithmetic of the quantiser's codes (one fused multiply-add with a per-block factor, the corrected quotient where 127
divides the maximum) restated in numpy and compared with the definition, RN_int(RN(x / RN(amax / 127))).  Every binary16
maximum: the subnormal ones, and every mantissa at the largest exponent -- a smaller exponent scales delta, r and x by the
same power of two, exactly, and leaves fewer values x."""
import numpy as np
import pytest

f32, f64 = np.float32, np.float64


def _quant_scale(amax):
    """delta, r and `refine` of a block; float32 scalars, every fused operation rounded once (its operands' products fit 53 bits)."""
    delta = amax / f32(127)
    r = f32(1) / delta
    half = f32(0.5) * amax
    fma = lambda a, b, c: f32(f64(a) * f64(b) + f64(c))  # noqa: E731
    up = fma(f32(-63.5), delta, half) >= f32(-2.0 ** -19) * delta
    side = fma(half, r, f32(-63.5))
    if up and side < 0:
        r = np.nextafter(r, f32(np.inf))
    if not up and side >= 0:
        r = np.nextafter(r, f32(0))
    refine = fma(f32(127), delta, -amax) == 0 or (fma(half, r, f32(-63.5)) >= 0) != up
    return delta, r, bool(refine)


def _codes(x, amax):
    delta, r, refine = _quant_scale(amax)
    if not refine:
        return np.rint(x.astype(f64) * f64(r))        # 1.5 * 2^23 is even: adding it rounds x r to an integer, ties to even
    q = (x * r).astype(f32)
    e = (x.astype(f64) - f64(delta) * q.astype(f64)).astype(f32)
    return np.rint((q.astype(f64) + e.astype(f64) * f64(r)).astype(f32))


def _check(amax_bits, lowest):
    n_refined = 0
    for bits in amax_bits:
        amax = np.array([bits], np.uint16).view(np.float16).astype(f32)[0]
        x = np.arange(max(0, lowest(bits)), bits + 1, dtype=np.uint16).view(np.float16).astype(f32)
        want = np.rint(x / (amax / f32(127)))
        assert want.max() == 127
        got = _codes(x, amax)
        assert np.array_equal(got, want), (bits, x[got != want][:4])
        n_refined += _quant_scale(amax)[2]
    return n_refined


def test_subnormal_maxima():
    assert _check(range(1, 1024), lambda bits: 0) == 8      # 127 divides the mantissa: 127, 254, ..., 1016


@pytest.mark.parametrize("part", range(4))
def test_every_mantissa(part):
    # values below 2^-9 of the maximum are below a quarter of delta: code 0 either way, one octave of them is looked at
    top = 30 << 10
    refined = _check(range(top + part * 256, top + (part + 1) * 256), lambda bits: bits - (10 << 10))
    assert refined == len([m for m in range(1024 + part * 256, 1024 + (part + 1) * 256) if m % 127 == 0])
