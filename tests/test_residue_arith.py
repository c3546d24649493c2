"""Host model of the residue products' arithmetic (csrc/rns.cu): the moduli, the FP32 reduction modulo p that
the operand conversion and the GEMM epilogue share, the 16-bit digits, and the reconstruction, against
exact integers. The constants come from the source, so a changed set of moduli is checked as it stands."""
import math
import os
import re

import numpy as np

SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                        "paper_1909_08596_gb300", "csrc", "rns.cu")).read()
MODS = [int(x) for x in re.search(r"constexpr int p\[kMods\] = \{([^}]*)\}", SRC).group(1).split(",")]
BETA = int(re.search(r"constexpr int kBeta = (\d+);", SRC).group(1))
SEG = 64 * int(re.search(r"constexpr int kSegStages = (\d+);", SRC).group(1))
F = np.float32


def sym_mod(v, p):
    """r = v - p rint(v / p) as the kernels form it: one fused multiply-add into 1.5 * 2^23 + v (1 / p)."""
    magic = np.float64(12582912)
    t = F(v.astype(np.float64) * np.float64(F(1) / F(p)) + magic)       # exact in FP64 before the one rounding
    return (v.astype(np.float64) - (t - F(magic)).astype(np.float64) * p).astype(np.int64)


def test_moduli():
    assert all(math.gcd(a, b) == 1 for i, a in enumerate(MODS) for b in MODS[:i])
    assert max(MODS) == 256 and 255 not in MODS
    assert math.prod(MODS) > 2 * 2 ** (2 * BETA)


def test_reduction_over_every_sum():
    """Every value an accumulator can hold before a reduction: a segment of products of residues plus the running
    residue. All stay below 2^24 (exact in FP32), and every reduced value fits a signed byte modulo p."""
    for p in MODS:
        lim = SEG * (p // 2) ** 2 + 128
        assert lim < 2 ** 24
        ends = [np.arange(-lim, -lim + 200000), np.arange(-200000, 200000), np.arange(lim - 200000, lim + 1)]
        mid = np.arange(-lim, lim + 1, 37)
        halves = (np.arange(-lim // p, lim // p)[:, None] * p + np.array([p // 2, p // 2 + 1])).ravel()
        for v in ends + [mid, halves[np.abs(halves) <= lim]]:
            r = sym_mod(v.astype(np.float32), p)
            assert not ((r - v) % p).any()
            assert np.abs(r).max() <= (128 if p == 256 else 127)


def test_digits_and_reconstruction():
    """A random product of scaled integers: residues from 16-bit digits, the products modulo p, and the integer
    back from them, for magnitudes up to the bound and for exact cancellation."""
    rng = np.random.default_rng(3)
    P = math.prod(MODS)
    W = [(P // p) * pow(P // p, -1, p) for p in MODS]

    def residues(a):
        b = a + 0x8000800080008000
        c = [((b >> (16 * j)) & 0xFFFF) - 0x8000 for j in range(4)]
        assert sum(x << (16 * j) for j, x in enumerate(c)) == a
        out = []
        for p in MODS:
            w = [pow(2, 16 * j, p) for j in range(4)]
            w = [x - p if x > p // 2 else x for x in w]
            v = sum(x * y for x, y in zip(c, w))
            assert abs(v) < 2 ** 24
            out.append(int(sym_mod(np.array([v], dtype=np.float32), p)[0]))
        return out

    for K in (1, 3, 40):
        for top in (10, 40, BETA - 3 - K.bit_length() // 2):
            a = [int(x) for x in rng.integers(-2 ** top, 2 ** top, K)]
            b = [int(x) for x in rng.integers(-2 ** top, 2 ** top, K)]
            if K == 40 and top == 10:
                a[-1], b[-1] = -sum(x * y for x, y in zip(a[:-1], b[:-1])), 1  # the product is exactly zero
            ra, rb = [residues(x) for x in a], [residues(x) for x in b]
            r = [sum(x[i] * y[i] for x, y in zip(ra, rb)) % p for i, p in enumerate(MODS)]
            x = sum(ri * wi for ri, wi in zip(r, W)) % P
            x = x - P if x > P // 2 else x
            assert x == sum(u * v for u, v in zip(a, b))
