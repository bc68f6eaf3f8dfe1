"""The 60-bit fixed-point dot products of the large-step double update (q60.cuh), emulated with Python
integers and checked against exact rational arithmetic: no sum leaves 64 bits, no limb leaves 32, and a
three-term complex dot product errs by less than 2^-57. CPU only."""
import random
import struct
from fractions import Fraction

import pytest


def to_lq(x):
    b = struct.unpack("<Q", struct.pack("<d", x))[0]
    ed = (b >> 52) & 0x7FF
    q = (((b & ((1 << 52) - 1)) | (1 << 52)) << 8) >> min((1023 - ed) & 0xFFFFFFFF, 63)
    h, l = q >> 30, q & 0x3FFFFFFF
    return (-h, -l) if b >> 63 else (h, l)


def dot(terms):
    hh = c = 0
    for (ah, al), (bh, bl) in terms:
        for limb in (ah, al, bh, bl):
            assert -(1 << 31) < limb < (1 << 31)
        hh += ah * bh
        c += ah * bl
        c += al * bh
        assert max(abs(hh), abs(c)) < 1 << 63
    v = hh + (c >> 30)
    assert -(1 << 63) <= v < (1 << 63) and -(1 << 31) <= v >> 30 < (1 << 31)
    return v


def unit(rng, kind):
    if kind == "axis":  # entries of magnitude 1, zeros and tiny numbers
        v = [0.0] * 6
        v[rng.randrange(6)] = rng.choice((1.0, -1.0, 1.0 - 2.0 ** -53))
        v[rng.randrange(6)] += rng.choice((0.0, 2.0 ** -59, 2.0 ** -80, 5e-324))
        return v
    v = [rng.gauss(0, 1) for _ in range(6)] if kind == "haar" else [rng.choice((-1.0, 1.0)) for _ in range(6)]
    n = sum(t * t for t in v) ** 0.5
    return [t / n for t in v]


@pytest.mark.parametrize("kind", ["haar", "equal", "axis"])
def test_dot_products(kind):
    rng = random.Random(60)
    worst = Fraction(0)
    for _ in range(3000):
        a, b = unit(rng, kind), unit(rng, rng.choice(("haar", kind)))
        v = dot([(to_lq(x), to_lq(y)) for x, y in zip(a, b)])
        worst = max(worst, abs(Fraction(v, 1 << 60) - sum(Fraction(x) * Fraction(y) for x, y in zip(a, b))))
    assert worst < Fraction(1, 1 << 57)


def test_conversion_truncates_toward_zero():
    rng = random.Random(61)
    for x in [0.0, 5e-324, 1.0, -1.0, 2.0 - 2.0 ** -52, 2.0 ** -60, 2.0 ** -61] + [rng.uniform(-2, 2) * 2.0 ** -rng.randrange(70) for _ in range(3000)]:
        h, l = to_lq(x)
        off = abs(Fraction(x)) - Fraction(abs((h << 30) + l), 1 << 60)
        assert 0 <= off < Fraction(1, 1 << 60)
