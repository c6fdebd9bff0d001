"""The conversions and shifts of the fixed-point code (csrc/qcs_ozaki.cuh, csrc/qcs_fixed.cuh) on
the CPU, over every exponent: the nearest integer, ties away from zero for the sliced entries
and upward for the shifts; entries far below the scale, and zeros, give zero."""
from __future__ import annotations

import ctypes
import random
from fractions import Fraction
from math import floor

import pytest

import warp_emulation

SOURCE = """
extern "C" long long host_fixed_of(double x, int e) { return qcs_oz::fixed_of(x, e); }
extern "C" long long host_fx_of1(double x, int f) { return fx_of1(x, f); }
extern "C" long long host_shift1(long long X, int s) { return fx_shift1(X, s); }
extern "C" long long host_scale(long long z, int g) { return qcs_oz::scale_of_fixed(z, g); }
extern "C" long long host_shift_any(long long X, int s) { return fx_shift_any(X, s); }
// a . b of two rows through the slices: z and its exponent
extern "C" long long host_sliced_dot(int n, const double *a, const double *b, int *exponent) {
    using namespace qcs_oz;
    int e[2] = {kNoRow, kNoRow};
    for (int k = 0; k < n; ++k) {
        if (a[k] != 0.0) e[0] = std::max(e[0], row_exp_of(a[k]));
        if (b[k] != 0.0) e[1] = std::max(e[1], row_exp_of(b[k]));
    }
    float acc[kLevels] = {};
    for (int k = 0; k < n; ++k) {
        const uint64_t u = (uint64_t)fixed_of(a[k], e[0]) + kDigitBias, v = (uint64_t)fixed_of(b[k], e[1]) + kDigitBias;
        for (int i = 1; i <= kSlices; ++i)
            for (int j = 1; i + j <= 8; ++j) acc[i + j - 2] += slice_f32(u, i) * slice_f32(v, j);  // exact in FP32
    }
    *exponent = e[0] + e[1] - 56;
    return combine_levels(acc);
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    lib = warp_emulation.compile_host(SOURCE, ["qcs_fixed.cuh"], str(tmp_path_factory.mktemp("emu")))
    for f in ("host_fixed_of", "host_fx_of1", "host_shift1", "host_scale", "host_shift_any"):
        getattr(lib, f).restype = ctypes.c_longlong
        getattr(lib, f).argtypes = [ctypes.c_double if "of" in f else ctypes.c_longlong, ctypes.c_int]
    lib.host_sliced_dot.restype = ctypes.c_longlong
    return lib


def mantissas(rng):
    return [1.0, 1.5, 2.0 - 2.0**-52, 1.0 + 2.0**-52] + [1.0 + rng.random() for _ in range(4)]


def test_conversions_round_to_nearest(host):
    """fixed_of for |x| (1 + 2^-7) < 2^e, fx_of1 for |x| 2^f < 2^62: half away from zero."""
    rng = random.Random(4)
    for k in range(-1000, 1):
        for m in mantissas(rng):
            for x in (m * 2.0**k, -m * 2.0**k):
                away = lambda v: (1 if v >= 0 else -1) * floor(abs(v) + Fraction(1, 2))
                e = 2
                assert host.host_fixed_of(x, e) == away(Fraction(x) * Fraction(2) ** (55 - e)), (x, e)
                f = 60
                assert host.host_fx_of1(x, f) == away(Fraction(x) * Fraction(2) ** f), (x, f)
    for x in (0.0, -0.0):
        assert host.host_fixed_of(x, 1) == 0 and host.host_fixed_of(x, 900) == 0 and host.host_fx_of1(x, 50) == 0


def test_shifts_round_to_nearest(host):
    """X 2^s for |X| < 2^62 and a result below 2^62: halves upward."""
    rng = random.Random(5)
    values = [0, 1, -1, 2, -2, 3, -3, (1 << 61) - 1, 1 << 61, -(1 << 61), (1 << 62) - 1, -(1 << 62) + 1]
    values += [rng.choice([1, -1]) * rng.randrange(1 << b) for b in range(1, 63)]
    for X in values:
        for s in list(range(-140, 62 - abs(X).bit_length() + 1)) + [-100000, -1 << 30]:
            exact = 0 if s < -200 else floor(Fraction(X) * Fraction(2) ** s + Fraction(1, 2))
            assert host.host_shift_any(X, s) == exact, (X, s)
            assert host.host_shift1(X, s) == exact, (X, s)


def test_scale_bounds_every_entry(host):
    """2^G lies above every |z| 2^g (1 + 2^-7), whichever entry has the largest g, so that the
    slices' integers z 2^{55 + g - G} fit 55 bits; and by at most three bits where the upper
    word decides."""
    rng = random.Random(6)
    zs = [s * ((1 << b) + d) for b in range(61) for d in (-1, 0, 1) for s in (1, -1)] + [rng.randrange(-(1 << 62), 1 << 62)
                                                                                        for _ in range(200)]
    for z in zs:
        for g in (-80, 0, 40):
            G = host.host_scale(z, g)
            if z == 0:
                assert G == -100000
                continue
            assert abs(z) * 129 < 128 << (G - g), (z, g)
            if abs(z) >> 33:
                assert abs(z) << 3 >= 1 << (G - g), (z, g)
    # an entry without an upper word whose exponent exceeds the others'
    for za, ga, zb, gb in ((1 << 55, -80, 1 << 21, 0), (1 << 55, 0, 1 << 26, 40)):
        G = max(host.host_scale(za, ga), host.host_scale(zb, gb))
        for z, g in ((za, ga), (zb, gb)):
            assert abs(z) * Fraction(2) ** (55 + g - G) < 1 << 55


@pytest.mark.parametrize("kind", ["uniform", "tiny", "top", "zeros"])
def test_sliced_dot(host, kind):
    """Within 2^-47 of the row scales: the entries' rounding (2^-56 each, 64 of them: 2^-50) and the
    dropped levels (level 9: 6 * 32 * 128^2 2^-70 = 2^-48.4, the others 2^-8 of it)."""
    rng = random.Random(8)
    for t in range(60):
        a = [rng.uniform(-1, 1) for _ in range(32)]
        b = [rng.uniform(-1, 1) * 2.0 ** rng.randrange(-4, 4) for _ in range(32)]
        if kind == "tiny":  # entries far below the scale, which must not leave a unit behind
            a = [x if k < 3 else x * 2.0 ** -rng.randrange(50, 200) for k, x in enumerate(a)]
        if kind == "top":  # digits at their bounds
            a = [rng.choice([1, -1]) * (1 - 2.0**-7 - 2.0**-20) for _ in a]
            b = [rng.choice([1, -1]) * (1 - 2.0**-7 - 2.0**-20) for _ in b]
        if kind == "zeros":
            b = [x if k % 5 == t % 5 else 0.0 for k, x in enumerate(b)]
        arr = ctypes.c_double * 32
        e = ctypes.c_int()
        z = host.host_sliced_dot(32, arr(*a), arr(*b), ctypes.byref(e))
        exact = sum(Fraction(x) * Fraction(y) for x, y in zip(a, b))
        scale = Fraction(2) ** (e.value + 56)
        assert abs(z * Fraction(2) ** e.value - exact) <= scale / 2**47
