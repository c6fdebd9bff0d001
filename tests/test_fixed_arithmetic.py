"""CPU model of the eliminations' fixed-point arithmetic (csrc/qcs_fixed.cuh).

An entry is a 64-bit integer X = h 2^31 + l with |l| <= 2^30; a product keeps
hh 2^62 + (h l' + l h') 2^31 and drops l l'; the complex pivot reciprocal is one third-order
step from a single-precision seed.  The bounds below are derived from the limb sizes:
the dropped term is at most 2^60 of a product of 2^121 (|X| < 2^60.5), and the reciprocal
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
    h = s32((X + (1 << 30)) >> 31)
    l = s32(X - (h << 31))
    assert X == (h << 31) + l and abs(l) <= 1 << 30
    return h, l


def mac(acc, a, b):
    acc[0] += a[0] * b[0]
    acc[1] += a[0] * b[1] + a[1] * b[0]
    assert abs(acc[0]) < 1 << 63 and abs(acc[1]) < 1 << 63  # what the 64-bit accumulators hold


def value(acc, up):
    v = (acc[0] << up) + (acc[1] >> (31 - up))
    assert abs(v) < 1 << 63
    return v


def inverse(qx, qy):
    """2^119 / (qx + i qy), as the device function."""
    a, b = split(qx), split(qy)
    s = [0, 0]
    mac(s, a, a)
    mac(s, b, b)
    D = s[0] + (s[1] >> 31)
    R0 = int(np.float32(np.float32(1) / np.float32(D >> 31)) * np.float32(2.0**54))
    e = s64(-(D * R0))
    eh = e >> 32
    e2 = (eh * eh) >> 32
    R = (R0 << 33) + ((R0 * eh) >> 20) + ((R0 * (e & 0xFFFFFFFF)) >> 52) + ((R0 * e2) >> 41)
    r = split(R)
    u, v = [0, 0], [0, 0]
    mac(u, a, r)
    mac(v, b, r)
    return value(u, 1), -value(v, 1)


def pivots(count, rng):
    for _ in range(count):
        q = [rng.randrange(-(1 << 61) + 1, 1 << 61), rng.randrange(-(1 << 61) + 1, 1 << 61)]
        k = rng.randrange(2)
        q[k] = rng.choice([1, -1]) * rng.randrange(1 << 60, 1 << 61)
        if rng.random() < 0.3:
            q[1 - k] >>= rng.randrange(62)
        yield q
    for x in (1 << 60, (1 << 61) - 1):
        for y in (0, 1, -1, 1 << 59, (1 << 61) - 1, -(1 << 61) + 1):
            yield [x, y]
            yield [y, -x]


def test_pivot_reciprocal():
    worst = 0.0
    for qx, qy in pivots(20000, random.Random(1)):
        ix, iy = inverse(qx, qy)
        n = qx * qx + qy * qy
        ex, ey = Fraction(qx << 119, n), Fraction(-qy << 119, n)
        err = float(max(abs(ix - ex), abs(iy - ey))) / float(max(abs(ex), abs(ey)))
        worst = max(worst, err)
    assert worst <= 2.0**-54


@pytest.mark.parametrize("bits_g,bits_v", [(59.5, 58), (59.5, 61), (40, 58), (59.5, 20)])
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
            assert abs(Fraction(value(acc, 3)) - Fraction(ex, 1 << 59)) <= 6
