"""The reflector scalars of the Householder steps in integers (hh_reflector in csrc/la.cuh on the
arithmetic of csrc/fx.cuh) and the reciprocal root of the Cholesky pivots, emulated with seeds off by
the error that rsqrt.approx and rcp.approx may have, against values of 60 digits."""
import math
import random
import struct
from decimal import Decimal, getcontext

import numpy as np
import pytest

getcontext().prec = 60
M64 = (1 << 64) - 1


def _hi(a, b):
    return (a * b) >> 64


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _to(x, s):
    """fx_to: 54 leading bits, the last one rounded up."""
    if x == 0:
        return 0.0
    a = abs(x)
    z = 64 - a.bit_length()
    n = (a << z) & M64
    return math.copysign(math.ldexp((n >> 11) + ((n >> 10) & 1), 11 - z + s), x)


def _rsqrt(s, err):
    y0 = int(min(float(np.float32(1 / math.sqrt(s / 2.0 ** 62))) * (1 + err) * 2.0 ** 32, 4294967040.0))
    e = (1 << 62) - _hi(s, y0 * y0)
    eh = e >> 20
    corr = (e >> 1) + ((3 * ((eh * eh) >> 22)) >> 3)
    return (y0 << 30) + _hi(corr << 18, y0 << 14)


def _rcp(u, err):
    r0 = int(float(np.float32(2.0 ** 64 / u)) * (1 + err) * 2.0 ** 29)
    e = (1 << 61) - _hi(u, r0 << 32)
    eh = e >> 20
    return (r0 << 26) + _hi((e + ((eh * eh) >> 21)) << 20, r0 << 9)


def _even(d):
    b = _bits(d)
    ex = ((b >> 52) & 0x7ff) - 1023
    odd = ex & 1
    return ((b & 0xfffffffffffff) | 1 << 52) << (10 + odd), (ex - odd) >> 1, 0 < b < 1 << 63 and -1000 <= ex <= 1000


def _reflector(d, xk, e1, e2):
    s, h, ok = _even(d)
    N = _hi(s, _rsqrt(s, e1))
    b = _bits(abs(xk))
    ex = b >> 52
    sig, expo = ((b & 0xfffffffffffff) | 1 << 52, ex - 1022) if ex else (0, -100000)
    sh = min(expo - 53 - h + 60, 9)
    V = N + (sig << sh if sh >= 0 else (sig >> -sh if sh > -63 else 0))
    zs = 11 - (64 - V.bit_length())
    dv = (((V >> (zs - 1)) + 1) >> 1 << zs) - V
    q = _hi((N + dv) << 2, V << 1)
    assert max((N + dv) << 2, V << 1) <= M64 and q > 0 and 2 <= zs <= 10
    z = 64 - q.bit_length()
    neg = math.copysign(1.0, xk) < 0 and xk != 0
    nrm = _to(N, h - 60)
    return ok, nrm, -nrm if neg else nrm, _to(-V if neg else V, h - 60), _to(_rcp(q << z, e2), z - 2 * h - 60)


def _values():
    rng = random.Random(5)
    for k in range(3000):
        scale = 2.0 ** rng.randint(-480, 480)
        x = [rng.gauss(0, 1) * 2.0 ** -rng.choice([0, 0, 3, 30, 70]) * scale for _ in range(rng.randint(1, 8))]
        d = 0.0
        for v in x:
            d += v * v
        if 2.0 ** -1000 <= d:
            yield d, x[0]
    for d, xk in ((1.0, 1.0), (1.0, -1.0), (4.0, 2.0), (3.9999999999999996, 1.9999999999999998), (2.0, 0.0), (2.0, -0.0),
                  (math.nextafter(4.0, 0.0), 0.0), (1.0, 5e-324), (2.0 ** -1000, 2.0 ** -500), (2.0 ** 1000, -2.0 ** 500)):
        yield d, xk


@pytest.mark.parametrize("sign", [-1, 0, 1])
def test_scalars_are_rounded_values(sign):
    e1, e2 = sign * 2.0 ** -22, -sign * 2.0 ** -22
    for d, xk in _values():
        ok, nrm, shift, vk, beta = _reflector(d, xk, e1, e2)
        assert ok
        root = Decimal(d).sqrt()
        # half a unit of the rounding, and at most 2^-58 before it
        half = Decimal(2) ** -53 * Decimal("1.04")
        assert abs(Decimal(nrm) / root - 1) <= half * 2, (d, xk)
        assert shift == (-nrm if xk < 0 else nrm)
        v = root + abs(Decimal(xk))
        assert abs(abs(Decimal(vk)) / v - 1) <= half * 2 and (vk < 0) == (xk < 0)
        # beta ||v||^2 = 2 for the v formed: 2^-54 of the reciprocal's last bit and the truncated product,
        # and the rounding
        v2 = Decimal(d) - Decimal(xk) ** 2 + Decimal(vk) ** 2
        assert abs(Decimal(beta) * v2 / 2 - 1) <= half * 2 + Decimal(2) ** -54, (d, xk)
        s, h, _ = _even(d)
        assert abs(Decimal(_to(_rsqrt(s, e1), -62 - h)) * root - 1) <= half * 2


def test_other_exponents_are_refused():
    for d in (0.0, 5e-324, 2.0 ** -1010, 2.0 ** 1010, math.inf, math.nan, -1.0):
        assert not _even(d)[2]


def test_entries_of_the_trailing_triangle():
    """wchol's row of a packed index, from a single-precision root with its error: every row of the
    largest trailing block with its border."""
    for K in (1, 2, 31, 47, 63):
        idx = 0
        for a in range(K + 1):
            for b in range(min(a + 1, K)):
                r = np.float32(8 * idx + 2)
                for err in (-2.0 ** -22, 0.0, 2.0 ** -22):
                    root = np.float32(r * np.float32(1 / math.sqrt(float(r)) * (1 + err)))
                    got = int((root - np.float32(1)) * np.float32(0.5))
                    assert (got, idx - got * (got + 1) // 2) == (a, b)
                idx += 1
        assert idx == K * (K + 1) // 2 + K
