"""The integer conversion of geometric factors to the fixed-point grid (fx_setup.cu), restated with Python integers:
the result to 2^-62 of itself plus half a unit, and the upper bound that fixes an element's exponent."""
import math
import random
import struct
from fractions import Fraction

M64, M32 = (1 << 64) - 1, (1 << 32) - 1


def _bits(g):
    u = struct.unpack("<Q", struct.pack("<d", abs(g)))[0]
    return u >> 52, (u & ((1 << 52) - 1)) | (1 << 52)


def _weight(r):
    """r > 0 as (m, x): m 2^(x-63) with 2^63 <= m < 2^64, m cut."""
    x = math.frexp(float(r))[1]
    m = int(r * Fraction(2) ** (64 - x))
    if m > M64:
        m, x = int(r * Fraction(2) ** (63 - x)), x + 1
    return m, x - 1


def _factor(g, f, k):
    ev, m53 = _bits(g)
    sh = 1023 + k - ev - f[1]
    p = ((m53 << 11) * f[0]) >> 64
    if ev == 0 or sh > 64:
        return 0
    r = p if sh <= 0 else ((p >> (sh - 1)) + 1) >> 1
    return -r if g < 0 else r


def _key(g, f):
    ev, m53 = _bits(g)
    p = (((m53 >> 32) << 11) * (f[0] >> 32)) >> 32
    up = p >> 31
    return 0 if ev == 0 else ((ev + f[1] - 1 + up) << 20) | ((p >> (10 + up)) & 0xFFFFF)


def _value(key):
    return Fraction((1 << 20) + (key & 0xFFFFF), 1 << 20) * Fraction(2) ** ((key >> 20) - 1022)


def _float32(x):
    return struct.unpack("<f", struct.pack("<f", x))[0]


def _key_sum(keys, top):
    e = top >> 20

    def rel(k):
        d = (k >> 20) - e
        return 0.0 if d < -60 else struct.unpack("<f", struct.pack("<I", ((127 + d) << 23) | ((k & 0xFFFFF) << 3)))[0]
    s = _float32(_float32(rel(keys[0]) + rel(keys[1])) + rel(keys[2]))
    return (struct.unpack("<I", struct.pack("<f", s))[0] >> 3) + ((e - 127) << 20) + 8


def test_conversion_and_bounds():
    rnd = random.Random(5)
    for _ in range(4000):
        scale = 2.0 ** rnd.randint(-150, 150)
        f = _weight(Fraction(rnd.uniform(1.0, 2.0)) / Fraction(rnd.uniform(1e-7, 1.0)))
        r = Fraction(f[0]) * Fraction(2) ** (f[1] - 63)
        g = [rnd.choice((-1, 1)) * scale * 2.0 ** -rnd.uniform(0, rnd.choice((1, 8, 70))) for _ in range(3)]
        keys = [_key(v, f) for v in g]
        for v, key in zip(g, keys):
            exact = abs(Fraction(v)) * r
            assert exact * (1 - Fraction(1, 1 << 18)) <= _value(key) <= exact
        total = sum(abs(Fraction(v)) for v in g) * r
        bound = _key_sum(keys, max(keys))
        assert total <= _value(bound) <= total * (1 + Fraction(1, 1 << 15))
        k = (bound >> 20) - 1021
        assert total < Fraction(2) ** k <= 4 * total
        for v in g:
            exact = Fraction(v) * r * Fraction(2) ** (62 - k)
            assert abs(_factor(v, f, k) - exact) <= Fraction(1, 2) + abs(exact) / (1 << 61)
    assert _factor(0.0, (1 << 63, 0), 0) == 0 and _key(0.0, (1 << 63, 0)) == 0
