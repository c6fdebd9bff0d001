"""CPU model of the eliminations' fixed-point arithmetic (csrc/qcs_fixed.cuh).

An entry is a 64-bit integer X = h 2^30 + l with |l| <= 2^29; a product keeps
hh 2^60 + (h l' + l h') 2^30 and drops l l'; the complex pivot reciprocal is one third-order
step from a single-precision seed.  The bounds below are derived from the limb sizes:
the dropped term is at most 2^58 of a product of 2^119 (|X| < 2^60), and the reciprocal
keeps at least 57 bits with at most four truncations of one unit each plus a seed error
e <= 2^-22, e^3 <= 2^-66.
"""
from __future__ import annotations

import random
from fractions import Fraction

import numpy as np
import pytest


def s64(x):
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >> 63 else x


def s32(x):
    x &= (1 << 32) - 1
    return x - (1 << 32) if x >> 31 else x


def split(X):
    h = s32((X + (1 << 29)) >> 30)
    l = s32(X - (h << 30))
    assert X == (h << 30) + l and abs(l) <= 1 << 29
    return h, l


def mac(acc, a, b):
    acc[0] += a[0] * b[0]
    acc[1] += a[0] * b[1] + a[1] * b[0]
    assert abs(acc[0]) < 1 << 63 and abs(acc[1]) < 1 << 63  # what the 64-bit accumulators hold


def value(acc, dn):
    v = (acc[0] << (60 - dn)) + (acc[1] >> (dn - 30))
    assert abs(v) < 1 << 63
    return v


def inverse(qx, qy):
    """2^118 / (qx + i qy), as the device function."""
    a, b = split(qx), split(qy)
    s = [0, 0]
    mac(s, a, a)
    mac(s, b, b)
    D = s[0] + (s[1] >> 30)
    R0 = int(np.float32(np.float32(1) / np.float32(D >> 31)) * np.float32(2.0**54))
    e = s64(-(D * R0))
    eh = e >> 32
    e2 = (eh * eh) >> 32
    R = (R0 << 33) + ((R0 * eh) >> 20) + ((R0 * (e & 0xFFFFFFFF)) >> 52) + ((R0 * e2) >> 41)
    r = split(R)
    u, v = [0, 0], [0, 0]
    mac(u, a, r)
    mac(v, b, r)
    return value(u, 60), -value(v, 60)


def pivots(count, rng):
    for _ in range(count):
        q = [rng.randrange(-(1 << 60) + 1, 1 << 60), rng.randrange(-(1 << 60) + 1, 1 << 60)]
        k = rng.randrange(2)
        q[k] = rng.choice([1, -1]) * rng.randrange(1 << 59, 1 << 60)
        if rng.random() < 0.3:
            q[1 - k] >>= rng.randrange(62)
        yield q
    for x in (1 << 59, (1 << 60) - 1):
        for y in (0, 1, -1, 1 << 58, (1 << 60) - 1, -(1 << 60) + 1):
            yield [x, y]
            yield [y, -x]


def test_pivot_reciprocal():
    worst = 0.0
    for qx, qy in pivots(20000, random.Random(1)):
        ix, iy = inverse(qx, qy)
        n = qx * qx + qy * qy
        ex, ey = Fraction(qx << 118, n), Fraction(-qy << 118, n)
        err = float(max(abs(ix - ex), abs(iy - ey))) / float(max(abs(ex), abs(ey)))
        worst = max(worst, err)
    assert worst <= 2.0**-54


@pytest.mark.parametrize("bits_g,bits_v", [(59.5, 58), (59.5, 60), (40, 58), (59.5, 20)])
def test_rank2_entry_update(bits_g, bits_v):
    """A + g_i v_j - v_i g_j with g scaled by 2^59: the dropped limb products and the two
    shifts cost at most 6 units of the result's last place."""
    rng = random.Random(2)
    lim = lambda b: rng.randint(-int(2.0**b) + 1, int(2.0**b) - 1)
    for _ in range(4000):
        g = [lim(bits_g) for _ in range(4)]
        v = [lim(bits_v) for _ in range(4)]
        S = [split(x) for x in g], [split(x) for x in v]
        neg = lambda t: (-t[0], -t[1])
        (gir, gii, gjr, gji), (vir, vii, vjr, vji) = S
        re, im = [0, 0], [0, 0]
        for a, b in ((gir, vjr), (neg(gii), vji), (neg(vir), gjr), (vii, gji)):
            mac(re, a, b)
        for a, b in ((gir, vji), (gii, vjr), (neg(vir), gji), (neg(vii), gjr)):
            mac(im, a, b)
        ere = g[0] * v[2] - g[1] * v[3] - v[0] * g[2] + v[1] * g[3]
        eim = g[0] * v[3] + g[1] * v[2] - v[0] * g[3] - v[1] * g[2]
        if max(abs(ere), abs(eim)) >= 1 << 121:
            continue  # beyond the bound 4 2^mb 2^59 that pivoting gives for |g| <= sqrt 2
        for acc, ex in ((re, ere), (im, eim)):
            assert abs(Fraction(value(acc, 59)) - Fraction(ex, 1 << 59)) <= 6


# ---- balanced slices of the tensor-core congruence (csrc/qcs_ozaki.cuh)

BIAS = 0x80808080808080


def row_exp(row):
    return max(((int(np.float64(abs(x)).view(np.int64)) + (1 << 46)) >> 52) - 1022 for x in row if x != 0.0)


def fixed(x, e):
    v = Fraction(float(x)) * Fraction(2) ** (55 - e)
    u = int(abs(v) + Fraction(1, 2))
    return -u if v < 0 else u


def digits(u):
    b = u + BIAS
    assert 0 <= b < 1 << 56
    return [((b >> (8 * (7 - i))) & 0xFF) - 128 for i in range(1, 8)]


def combine(acc):
    """The level sums through the magic FP32 addition, modulo 2^64."""
    magics = [12582912.0] * 6 + [12582944.0]
    x = [int(np.float32(np.float32(a) + np.float32(m)).view(np.uint32)) for a, m in zip(acc, magics)]
    magic = 0x4B400000
    off = magic * 0x0000040404040404 + (magic >> 6)
    z = 4 * x[5] + (x[6] >> 6) + (x[4] << 10) + (x[3] << 18) + (x[2] << 26)
    z += ((x[0] * 1024 + x[1] * 4) & 0xFFFFFFFF) << 32
    return s64(z - off)


def sliced_dot(a, b):
    ea, eb = row_exp(a), row_exp(b)
    da, db = [digits(fixed(x, ea)) for x in a], [digits(fixed(x, eb)) for x in b]
    acc = []
    for L in range(2, 9):
        t = sum(da[k][i - 1] * db[k][L - i - 1] for i in range(1, 8) if 1 <= L - i <= 7 for k in range(len(a)))
        assert abs(t) < 1 << 22  # what the FP32 accumulators and the magic addition hold exactly
        acc.append(t)
    z = combine(acc)
    assert z == sum(acc[L - 2] << (8 * (7 - L) + 2) for L in range(2, 8)) + ((acc[6] + 32) >> 6)
    return Fraction(z) * Fraction(2) ** (ea + eb - 56), ea, eb


@pytest.mark.parametrize("scale", [1.0, 2.0**-30, 1.0 - 2.0**-53, 3.0])
def test_balanced_slices_reach_an_fp64_product(scale):
    """Digits reproduce the rounded entry, level sums stay below 2^22, and the dot product's
    error is within 2^-50 of the row scales: K = 32 entries with 2^-56 rounding each side
    (2 * 32 * 2^-56) and the dropped levels (at most 6 * 32 * 128^2 2^{-72+16} = 2^-34.4 2^{-16}
    per scale product, halved by the digits' signs)."""
    rng = np.random.default_rng(3)
    for t in range(60):
        a, b = rng.uniform(-1, 1, 32) * scale, rng.uniform(-1, 1, 32)
        if t % 3 == 0:
            a[rng.integers(32)] = scale  # an entry at the top of the scale
        if t % 4 == 0:
            b = np.where(np.arange(32) == t % 32, -1.0, 0.0)
        e = row_exp(a)
        for x in a:
            u = fixed(x, e)
            assert sum(d << (8 * (7 - i)) for i, d in enumerate(digits(u), 1)) == u
        got, ea, eb = sliced_dot(a, b)
        exact = sum(Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b))
        assert abs(got - exact) <= Fraction(2) ** (ea + eb - 47)


def test_largest_digits_accumulate_exactly():
    a = np.full(32, 1.0 - 2.0**-7 - 2.0**-20)
    for b in (a, -a):
        got, ea, eb = sliced_dot(a, b)
        exact = sum(Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b))
        assert abs(got - exact) <= Fraction(2) ** (ea + eb - 47)
