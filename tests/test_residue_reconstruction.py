"""Host model, operation by operation, of how csrc/rns.cu rebuilds a product from its residues (crt_fraction,
crt_offset, frac_add, frac_fold, crt_value): 32-bit words that wrap, the fold to a 64-bit fraction of P, the
multiplication by P's leading word, the rounding to 53 bits and the exponent; against exact integers.

Bound: the fraction is off by the rounding of its constants, at most sum |r_i| |c_i - exact|, and half of its last bit;
times P, absolute. Then P's truncated word, the truncated high product and the rounding to 53 bits, together
2^-53 (1 + 2^-8) of the result."""
import math
import os
import random
import re
import struct
from fractions import Fraction

import pytest

SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                        "paper_1909_08596_gb300", "csrc", "rns.cu")).read()
MODS = [int(x) for x in re.search(r"constexpr int p\[kMods\] = \{([^}]*)\}", SRC).group(1).split(",")]
BETA = int(re.search(r"constexpr int kBeta = (\d+);", SRC).group(1))
LIMB = int(re.search(r"kLimb = (\d+), kFrac = 32 \+ 2 \* kLimb;", SRC).group(1))
FRAC = 32 + 2 * LIMB
P = math.prod(MODS)
M32, M64 = 2 ** 32 - 1, 2 ** 64 - 1


def inverse(p):
    return pow(P // p % p, -1, p)


C = [((inverse(p) << FRAC) + p // 2) // p for p in MODS]
OFFSET = (-sum(128 * c for c in C) + (1 << (FRAC - 65))) % (1 << FRAC)


def words(x):
    return [x & (2 ** LIMB - 1), (x >> LIMB) & (2 ** LIMB - 1), x >> (2 * LIMB)]


def fraction(residues):
    """frac_start, frac_add over the moduli, frac_fold: bytes r in [-128, 127] to a 64-bit fraction of P."""
    w = words(OFFSET)
    for r, c in zip(residues, C):
        u = (r & 0xFF) ^ 0x80
        for j in range(3):
            w[j] += u * words(c)[j]
    assert w[0] <= M32 and w[1] <= M32          # only the top word wraps (modulo 1)
    w[2] &= M32
    m = w[1] + (w[0] >> LIMB)
    assert m <= M32
    t = (w[2] + (m >> LIMB)) & M32
    mask = 2 ** LIMB - 1
    return (t << 32) | (((m & mask) << (32 - LIMB)) & M32) | ((w[0] & mask) >> (2 * LIMB - 32))


def value(f, s):
    """crt_value: x 2^-s from f = 2^64 x / P."""
    p64 = P >> 54
    neg = f >> 63
    a = (-f) & M64 if neg else f
    lz = 64 - (a | 1).bit_length()
    h = (((a << lz) & M64) * p64) >> 64
    e = 63 + 54 - lz - s
    if not h >> 63:
        h = (h << 1) & M64
        e -= 1
    r = (h >> 11) + ((h >> 10) & 1)
    if not 0 <= e + 1021 <= 2043:               # scaled_value
        assert r <= 2 ** 53
        try:
            d = math.ldexp(float(r), e - 52)
        except OverflowError:
            d = math.inf
        return -d if neg else d
    hi = ((r >> 32) + ((e + 1022) << 20)) & M32
    d = struct.unpack("<d", struct.pack("<Q", (hi << 32) | (r & M32)))[0]
    return (-d if neg else d) if a else 0.0


def residues(x, rng=None):
    """Symmetric residues as the kernels keep them: |r| <= (p + 1) / 2, either neighbour where both fit a byte."""
    out = []
    for p in MODS:
        r = x % p
        r = r - p if r > p // 2 else r
        if rng and abs(r) >= p // 2 - 1 and rng.random() < 0.5:
            o = r - p if r > 0 else r + p
            r = o if abs(o) <= (p + 1) // 2 else r
        out.append(r if r <= 127 else r - 256)  # (128 as a byte, modulo 256)
    return out


FRACTION_ERROR = sum(Fraction(abs(c * p - (inverse(p) << FRAC)), p) * 128 for c, p in zip(C, MODS)) / 2 ** FRAC \
    + Fraction(1, 2 ** 65)
ABS = FRACTION_ERROR * P


def check(x, s, rng=None):
    v = value(fraction(residues(x, rng)), s)
    exact = Fraction(x) / (Fraction(2) ** s)
    tol = (Fraction(abs(x)) * (1 + Fraction(1, 256)) / 2 ** 53 + ABS * (1 + Fraction(1, 256))) / (Fraction(2) ** s)
    if abs(exact) < Fraction(2) ** -1020:
        tol += Fraction(1, 2 ** 1074)
    assert abs(Fraction(v) - exact) <= tol, (x, s, v)


def test_fraction_error_is_as_stated():
    bits = float(re.search(r"fraction is good to 2\^-([\d.]+) of P", SRC).group(1))
    assert FRACTION_ERROR <= Fraction(2.0 ** -bits)
    assert ABS / 2 ** (2 * BETA) <= Fraction(2.0 ** -float(
        re.search(r"that is\s+(?://\s*)?to 2\^-([\d.]+) of the product of the two rows' norm bounds", SRC).group(1)))


def test_zero_is_exact():
    assert value(fraction(residues(0)), 0) == 0.0
    for s in (-(1 << 12), 1 << 12):
        assert value(fraction(residues(0)), s) == 0.0


@pytest.mark.parametrize("top", [1, 2, 40, 53, 54, 64, 80, 100, 115, 116])
def test_random(top):
    rng = random.Random(top)
    for _ in range(400):
        x = rng.randrange(-(1 << top), (1 << top) + 1)
        check(x, rng.choice([0, 116, -300, 500]), rng)


def test_edges():
    """The largest products, carries out of 53 bits (all ones before the rounding), powers of two, and sums one step
    on either side of a residue's end."""
    rng = random.Random(1)
    big = 1 << (2 * BETA)
    xs = [0, 1, big, big - 1, big + (big >> 40)]
    xs += [(1 << k) + d for k in range(50, 2 * BETA) for d in (-1, 0, 1, -(1 << max(0, k - 54)), -(1 << max(0, k - 53)))]
    for p in MODS:
        xs += [p * rng.randrange(1 << 100) + d for d in (p // 2 - 1, p // 2, p // 2 + 1)]
    for x in xs:
        for y in (x, -x):
            check(y, 0, rng)


@pytest.mark.parametrize("residue", [127, -127, -128])
def test_every_residue_at_an_end(residue):
    """All bytes at an end of their range (the 20-bit words' largest and smallest sums), whatever integer that is."""
    r = [residue] * len(MODS)
    x = sum(v * inverse(p) * (P // p) for v, p in zip(r, MODS)) % P
    x = x - P if x > P // 2 else x
    f = fraction(r)
    f = f - 2 ** 64 if f >> 63 else f
    d = Fraction(f, 2 ** 64) - Fraction(x, P)
    assert min(abs(d), abs(abs(d) - 1)) <= FRACTION_ERROR


@pytest.mark.parametrize("s", [116 + 1000, 116 + 1022, 116 + 1040, 116 + 1074, 116 + 1090, 116 - 1020, 116 - 1023])
def test_ends_of_the_exponent_range(s):
    rng = random.Random(s)
    for _ in range(200):
        x = rng.randrange(1 << 110, 1 << 116)
        v = value(fraction(residues(x)), s)
        if Fraction(x) / Fraction(2) ** s >= Fraction(2) ** 1024:
            assert v == math.inf
        else:
            check(x, s)
