"""The longest sum of limb products, A' of the local energy (csrc/qcs_energy.cu), on the CPU at the
entries that make its 64-bit parts largest: every limb of a factor at its bound, all products of
one sign.  Parts modulo 2^64, the value compared with the exact one (the dropped products of
the lower limbs, a quarter of a unit each, and one unit of rounding)."""
from __future__ import annotations

import ctypes

import pytest

import warp_emulation

SOURCE = r"""
static int bits_of(int n) { return fx_ap_bits(n); }
// entries of b bits with both limbs at their bounds and of opposite signs
template <int S>
static fxl part(int b, int sign) {
    return fx_split<S>(sign > 0 ? (1ll << b) - (1ll << (S - 1)) : -(1ll << b) + (1ll << (S - 1)) - 1);
}
template <int S>
static int4 entry(int b, int sr, int si) {
    return fx_pack(part<S>(b, sr), part<S>(b, si));
}
static long long whole(int4 q, int S, bool im) { return im ? ((long long)q.z << S) + q.w : ((long long)q.x << S) + q.y; }
// A'_ab of the occupied block: 2n columns of K_a M_b - K_b M_a, as the kernel forms it
extern "C" int host_ap(int n, int bits, double *err) {
    fxacc p1 = {0, 0}, p2 = {0, 0}, p3 = {0, 0};
    __int128 re = 0, im = 0;
    *err = 0;
    for (int which = 0; which < 2; ++which) {  // the real part largest, then the imaginary one
        p1 = p2 = p3 = {0, 0};
        re = im = 0;
        for (int mu = 0; mu < 2 * n; ++mu) {
            const int4 x = entry<kFxS>(bits, 1, 1), y = entry<kFxS>(bits, 1, which ? 1 : -1);
            const int4 k = entry<kFxS>(bits, -1, -1), w = make_int4(-k.x, -k.y, -k.z, -k.w), z = y;
            for (int h = 0; h < 2; ++h) {
                const int4 a = h ? w : x, b = h ? z : y;
                fx_mac(p1, fx_re(a), fx_re(b));
                fx_mac(p2, fx_im(a), fx_im(b));
                fx_mac(p3, fx_add(fx_re(a), fx_im(a)), fx_add(fx_re(b), fx_im(b)));
                const __int128 ar = whole(a, kFxS, 0), ai = whole(a, kFxS, 1), br = whole(b, kFxS, 0), bi = whole(b, kFxS, 1);
                re += ar * br - ai * bi;
                im += ar * bi + ai * br;
            }
        }
        fxacc r = fx_accsub(p1, p2), i = fx_accsub(fx_accsub(p3, p1), p2);
        r.cr += fx_half<kFxS>(58);
        i.cr += fx_half<kFxS>(58);
        *err = std::max(*err, std::fabs((double)(fx_value<kFxS>(r, 58) - (long long)(re >> 58))));
        *err = std::max(*err, std::fabs((double)(fx_value<kFxS>(i, 58) - (long long)(im >> 58))));
    }
    return 0;
}
extern "C" int host_ap_bits(int n) { return bits_of(n); }
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return warp_emulation.compile_host(SOURCE, ["qcs_fxcong.cuh"], str(tmp_path_factory.mktemp("emu")))


@pytest.mark.parametrize("n", range(2, 25))
def test_operator_sums_stay_in_64_bits(host, n):
    err = ctypes.c_double()
    host.host_ap(n, host.host_ap_bits(n), ctypes.byref(err))
    # 8 products a column; a dropped l l' is below 2^56 in units of 2^58, so a quarter each
    assert err.value <= 2 * n * 8 / 4 + 1


def test_one_more_bit_would_not(host):
    """The test's entries do reach the bound: with 56 bits at n = 24 the sum leaves 64 bits."""
    err = ctypes.c_double()
    host.host_ap(24, 56, ctypes.byref(err))
    assert err.value > 1e9
