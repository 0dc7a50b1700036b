"""The integer arithmetic of csrc/fx.cuh, restated in Python integers and checked against its bounds:
limbs, sums of limb products, the reciprocal square root and the reciprocal from seeds of 22 bits."""
import math
import random
from fractions import Fraction

import numpy as np

B = 29


def split2(x):
    h = (x + (1 << (B - 1))) >> B
    return [x - (h << B), h]


def split4(x):
    half, mask = 1 << (B - 1), (1 << B) - 1
    y = x + (half << (2 * B)) + (half << B) + half
    return [(y & mask) - half, ((y >> B) & mask) - half, ((y >> (2 * B)) & mask) - half, y >> (3 * B)]


def join(w):
    return sum(v << (B * k) for k, v in enumerate(w))


def acc42(pairs, s):
    """FxAcc: sums of four-limb by two-limb products without the lowest pair, times 2^-s."""
    c = [0, 0, 0, 0]
    for p, a in pairs:
        c[3] += p[3] * a[1]
        c[2] += p[3] * a[0] + p[2] * a[1]
        c[1] += p[2] * a[0] + p[1] * a[1]
        c[0] += p[1] * a[0] + p[0] * a[1]
    assert all(abs(v) < 1 << 63 for v in c)
    if s == 60:
        return (c[3] << 56) + (c[2] << 27) + ((c[1] + (c[0] >> B) + 2) >> 2)
    return (c[3] << (116 - s)) + (c[2] << (87 - s)) + (c[1] << (58 - s)) + (c[0] >> (s - 29))


def acc44(pairs):
    c = [0, 0, 0, 0]
    for a, b in pairs:
        for i in range(4):
            for j in range(4):
                if i + j >= 3:
                    c[i + j - 3] += a[i] * b[j]
    assert all(abs(v) < 1 << 63 for v in c)
    return (c[3] << 62) + (c[2] << 33) + (c[1] << 4) + (c[0] >> 25)


def test_limbs_hold_every_value_and_stay_in_range():
    rng = random.Random(1)
    for bits in (0, 1, 28, 29, 57, 58, 86, 87, 114, 117):
        for x in [(1 << bits) - 1, -(1 << bits), 1 << bits] + [rng.randrange(-(1 << bits), 1 << bits) for _ in range(200)]:
            w = split4(x)
            assert join(w) == x
            assert all(-(1 << 28) <= v < 1 << 28 for v in w[:3]) and abs(w[3]) < 1 << 31
            if bits <= 58:
                assert join(split2(x)) == x


def test_product_sums_of_33_full_entries_fit_and_are_exact_to_their_bound():
    """|P| <= 2^114, |A| <= 2^57, 33 terms: no accumulator overflows, errors below 2^-109 and 2^-108."""
    rng = random.Random(2)
    for trial in range(60):
        def full(k):
            return rng.choice([-1, 1]) * ((1 << k) - (rng.randrange(1 << 20) if trial % 2 else rng.randrange(1 << k)))
        P, A = [full(114) for _ in range(33)], [full(57) for _ in range(33)]
        if trial == 0:
            P, A = [1 << 114] * 33, [1 << 57] * 33
        exact = sum(p * a for p, a in zip(P, A))
        for s in (54, 55, 57, 60):
            got = acc42([(split4(p), split2(a)) for p, a in zip(P, A)], s)
            assert abs(Fraction(exact, 1 << s) - got) <= 40, (s, trial)
        L, Y = [full(113) for _ in range(16)], [full(114) for _ in range(16)]
        got = acc44([(split4(x), split4(y)) for x, y in zip(L, Y)])
        assert abs(Fraction(sum(x * y for x, y in zip(L, Y)), 1 << 112) - got) <= 1 << 9


def _hi(a, b):
    return (a * b) >> 64


def test_reciprocal_square_root_and_reciprocal_from_seeds():
    rng = random.Random(3)
    edge = [1 << 62, (1 << 64) - 1, (1 << 63) - 1, (1 << 62) + 1]
    for s in edge + [rng.randrange(1 << 62, 1 << 64) for _ in range(4000)]:
        m = s / 2.0 ** 62
        err = 1 + rng.uniform(-2, 2) * 2.0 ** -22  # rsqrt.approx: 2^-22.4
        y0 = int(min(float(np.float32(1 / math.sqrt(m))) * err * 2.0 ** 32, 4294967040.0))
        e = (1 << 62) - _hi(s, y0 * y0)
        eh = e >> 20
        corr = (e >> 1) + ((3 * ((eh * eh) >> 22)) >> 3)
        assert abs(corr << 18) < 1 << 63
        y = (y0 << 30) + _hi(corr << 18, y0 << 14)
        # y^2 m = 1 to 2^-58, so y to 2^-59
        assert abs(Fraction(y * y * s, 1 << 186) - 1) < Fraction(1, 1 << 58)
        # the same s as m = s 2^-64 in [1/4, 1)
        r0 = int(float(np.float32(4 / m)) * (1 + rng.uniform(-2, 2) * 2.0 ** -23) * 2.0 ** 29)
        e = (1 << 61) - _hi(s, r0 << 32)
        eh = e >> 20
        corr = e + ((eh * eh) >> 21)
        assert abs(corr << 20) < 1 << 63
        g = (r0 << 26) + _hi(corr << 20, r0 << 9)
        assert abs(Fraction(g * s, 1 << 119) - 1) < Fraction(1, 1 << 53)
