"""The integer contractions of the FP64 operator (csrc/nsk_fx.cuh), restated in Python integers and
compared with exact rational sums: the fixed-point limbs, the three-product sum and the rounding of
the result, over line lengths, magnitudes, signs and exceptional values.

Bound, derived from the representation before any run: a line's values lose less than 2^4 units of
2^(E - 1023 - 61) each (the bits below the low limb; the shift and the one's complement of a negative
value lie inside them); value pairs are added and subtracted exactly; the matrix entries (half sums and
half differences) are off by at most 2^3 units of 2^(es - 1023 - 61) (rounded to 2^4). In units of the
sum (2^64 of the product's): pairs below 2^63 times entry errors of 2^3, W entries: 4 W; pair errors
below 2^5 times entries whose magnitudes add up to less than 2^62: 8; each low-low product below 2 units:
2 W; two floors: 2. Together at most 10 (W + 1) units, and the rounding to FP64 adds half an ulp of the
result."""
import math
from fractions import Fraction

import numpy as np
import pytest

M32 = 0xFFFFFFFF


def _words(x):
    b = int(np.float64(x).view(np.uint64))
    return b >> 32, b & M32


def _s32(v):
    return v - (1 << 32) if v & 0x80000000 else v


def _biased(s):
    return 0 if not s > 0.0 else max(math.frexp(s)[1] + 1022, 0)


def _entry(x, es):
    v = round(math.ldexp(x, 57 + 1023 - es))
    return v >> 28, v & 0xFFFFFFF


def _val(x, E):
    hi, lo = _words(x)
    sh = (E - (hi & 0x7FFFFFFF)) >> 20
    vh = (((hi << 9) | (lo >> 23)) & 0x1FFFFFFF) | 0x20000000
    v = ((vh << 32) | ((lo << 9) & M32)) >> sh if sh < 64 else 0
    s = M32 if hi >> 31 else 0
    return _s32((v >> 32) ^ s), ((v & M32) ^ s) >> 4


def _line(xs, row, es):
    """(sum, E): the row's sum at the line's exponent, from the sums and differences of value pairs."""
    E = max([100 << 20] + [_words(x)[0] & 0x7FFFFFFF for x in xs]) | 0xFFFFF
    v = [_val(x, E) for x in xs]
    W, total = len(xs), 0
    for sign in (-1, 1):
        hh = cr = 0
        for j in range(W // 2 + (W % 2 if sign > 0 else 0)):
            k = W - 1 - j
            if j == k:
                (h, low), (th, tl) = v[j], _entry(row[j], es)
            else:
                h, low = v[j][0] + sign * v[k][0], v[j][1] + sign * v[k][1]
                th, tl = _entry((row[j] + sign * row[k]) / 2, es)
            assert -(1 << 31) <= h < 1 << 31 and abs(low) < 1 << 29 and abs(th) <= 1 << 30 and 0 <= tl < 1 << 28
            hh += h * th
            cr += h * tl + low * th
        assert abs(hh) < 1 << 62 and abs(cr) < 1 << 62
        total += hh + (cr >> 28)
    return total, E


def _out(a, e):
    s = a < 0
    m = abs(a)
    lz = 64 - m.bit_length()
    m = (m << (lz & 63)) & ((1 << 64) - 1)
    r = (m >> 11) + ((m >> 10) & 1)
    eb = e - 1019 - lz
    if eb >= 2046:
        return math.nan
    if m == 0 or eb < 0:
        return 0.0
    bits = (r + (eb << 52)) | (int(s) << 63)
    return float(np.uint64(bits).view(np.float64))


def _contract(xs, row, es):
    a, E = _line(xs, row, es)
    ex = E >> 20
    return _out(a, ex + es + (65536 if ex >= 0x7FF else -65536 if ex <= 100 else 0)), ex


@pytest.mark.parametrize("W", [3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("spread", [0.0, 8.0, 60.0, 400.0])
def test_line_sum_within_the_derived_bound(W, spread):
    rng = np.random.default_rng(int(W * 1000 + spread))
    for _ in range(300):
        xs = rng.standard_normal(W) * 2.0 ** rng.uniform(-spread, spread, size=W)
        xs[rng.random(W) < 0.1] = 0.0
        row = rng.standard_normal(W) * 2.0 ** rng.uniform(-4, 12)
        es = _biased(float(np.abs(row).sum()) * rng.uniform(1.0, 3.0))  # the table's largest row, at least this one
        got, ex = _contract([float(x) for x in xs], [float(t) for t in row], es)
        want = sum(Fraction(float(x)) * Fraction(float(t)) for x, t in zip(xs, row))
        unit = Fraction(2) ** (max(ex, 100) + es - 2104)
        assert abs(Fraction(got) - want) <= 10 * (W + 1) * unit + abs(want) * Fraction(1, 2 ** 53)


@pytest.mark.parametrize("W", [5, 6, 8])
def test_smaller_error_than_fp64_accumulation(W):
    """Root mean square error over random lines below that of the FP64 fused multiply-add chain."""
    rng = np.random.default_rng(W)
    e_fx = e_fp = 0.0
    for _ in range(1000):
        xs, row = rng.uniform(-1, 1, W) + 1.0, rng.uniform(-8, 8, W)
        row[-1] = -row[:-1].sum()  # a cancelling operator, as a derivative of a smooth field
        want = sum(Fraction(float(x)) * Fraction(float(t)) for x, t in zip(xs, row))
        got, _ = _contract([float(x) for x in xs], [float(t) for t in row], _biased(float(np.abs(row).sum())))
        acc = Fraction(0)
        for x, t in zip(xs, row):  # one rounding per multiply-add
            acc = Fraction(float(acc + Fraction(float(x)) * Fraction(float(t))))
        e_fx += float(Fraction(got) - want) ** 2
        e_fp += float(acc - want) ** 2
    assert e_fx < e_fp


def test_exceptional_values():
    row, es = [1.0, -2.0, 0.5], _biased(3.5)
    assert _contract([0.0, -0.0, 0.0], row, es)[0] == 0.0
    assert math.isnan(_contract([1.0, math.inf, 0.0], row, es)[0])
    assert math.isnan(_contract([1.0, math.nan, 0.0], row, es)[0])
    assert _contract([5e-324, 1e-310, 2e-308], row, es)[0] == 0.0
    big = _contract([1e308, 1e308, 1e308], [1.0, 1.0, 1.0], _biased(3.0))[0]
    assert math.isnan(big) or math.isinf(big)  # overflow is not a finite value
