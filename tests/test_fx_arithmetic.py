"""The integer arithmetic of the FP64 tensor-core contraction, restated with
Python integers: digits of FP64 numbers, exactness of the levels, and the
joining of eight levels into one correctly rounded FP64 number."""
import math
import struct
from fractions import Fraction

import numpy as np
import pytest

MASK = (1 << 64) - 1


def bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def digits(x, M):
    """Eight balanced base-256 digits of x / 2^(M - 1022) at 62 fractional bits."""
    b = bits(x)
    e = (b >> 52) & 0x7FF
    m = ((b & ((1 << 52) - 1)) | (1 << 52)) << 9
    m = m >> (M - e) if 0 <= M - e < 64 else 0
    X = -m if b >> 63 else m
    Y = (X + 0x8080808080808080) & MASK
    return [((Y >> (8 * (7 - p))) & 255) - 128 for p in range(8)], X


def join(i, me):
    hi = (i[0] * 256 + i[1]) * 65536 + i[2] * 256 + i[3]
    lo = i[4] * 16777216 + i[5] * 65536 + i[6] * 256 + i[7]
    hi += lo >> 32
    l = lo & 0xFFFFFFFF
    sg = hi < 0
    ul = ((l ^ 0xFFFFFFFF) + 1) if sg else l
    uh = ((hi ^ -1) if sg else hi) + (ul >> 32)
    h1, h0, l = uh >> 32, uh & 0xFFFFFFFF, ul & 0xFFFFFFFF
    for _ in range(2):
        if h1 == 0:
            h1, h0, l, me = h0, l, 0, me - 32
    if h1 == 0:
        return 0.0
    z = 32 - h1.bit_length()
    m = (((h1 << 64 | h0 << 32 | l) << z) >> 32) & MASK
    be = me - z
    out = ((be - 1) << 52) + (m >> 11) + ((m >> 10) & 1)
    return struct.unpack("<d", struct.pack("<Q", out | (sg << 63)))[0]


@pytest.mark.parametrize("spread", [0, 20, 60, 300])
def test_digits_hold_62_bits_of_the_largest_entry(spread):
    rng = np.random.default_rng(spread)
    x = rng.standard_normal(200) * 2.0 ** rng.integers(-spread, spread + 1, 200)
    x[:3] = 0.0, -x.max(), np.nextafter(np.abs(x).max(), 0.0)
    M = max((bits(v) >> 52) & 0x7FF for v in x)
    for v in x:
        d, X = digits(v, M)
        assert all(-128 <= k <= 127 for k in d) and abs(d[0]) <= 64
        assert sum(k * 256 ** (7 - p) for p, k in enumerate(d)) == X
        err = Fraction(v) - Fraction(X) * Fraction(2) ** (M - 1022 - 62)
        assert abs(err) < Fraction(2) ** (M - 1022 - 62)


@pytest.mark.parametrize("N", [1, 64, 96, 128])
def test_levels_stay_exact_in_fp32(N):
    """The largest level 0..7 is below 2^24, so FP32 sums of its integers are exact in any order."""
    top = [64] + [128] * 7
    assert max(sum(top[p] * top[k - p] for p in range(k + 1)) * N for k in range(8)) < 1 << 24
    # the 32-bit partial joins of the two highest level pairs
    big = [sum(top[p] * top[k - p] for p in range(k + 1)) * N for k in range(8)]
    assert big[0] * 256 + big[1] < 1 << 31 and big[2] * 256 + big[3] < 1 << 31


@pytest.mark.parametrize("scale", [0, 1, 7])
def test_join_rounds_once(scale):
    rng = np.random.default_rng(scale)
    for _ in range(400):
        keep = rng.integers(0, 9)  # how many leading levels cancel
        i = [0 if k < keep else int(rng.integers(-(1 << 22 - scale), 1 << 22 - scale)) for k in range(8)]
        S = sum(v * 256 ** (7 - k) for k, v in enumerate(i))
        got = join(i, 1023 + 95)  # the sum as an integer
        assert Fraction(got) == S or abs(Fraction(got) - S) <= Fraction(math.ulp(float(S))) / 2


def test_dot_product_is_closer_than_a_multiply_add_chain():
    rng = np.random.default_rng(3)
    worse = 0
    for _ in range(50):
        a, t = rng.standard_normal(96) * 0.9 ** np.arange(96), rng.standard_normal(96)
        Ma, Mt = (max((bits(v) >> 52) & 0x7FF for v in x) for x in (a, t))
        da, dt = ([digits(v, M)[0] for v in x] for x, M in ((a, Ma), (t, Mt)))
        lev = [sum(da[n][p] * dt[n][k - p] for n in range(96) for p in range(k + 1)) for k in range(8)]
        exact = sum(Fraction(x) * Fraction(y) for x, y in zip(a, t))
        chain = 0.0
        for x, y in zip(a, t):
            chain = float(Fraction(x) * Fraction(y) + Fraction(chain))  # one rounding per term, as FMA
        w = join(lev, Ma + Mt - 994)
        worse += abs(Fraction(w) - exact) > max(abs(Fraction(chain) - exact), Fraction(math.ulp(float(exact))))
    assert worse == 0
