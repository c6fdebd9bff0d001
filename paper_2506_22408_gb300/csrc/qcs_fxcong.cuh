// qcs_fxcong.cuh -- the congruence of one pair in fixed point on the integer pipe: T (or
// K = Ut [H1 | G2]) from a walker's rows and a snapshot's, and B^(s) from it, for the kernels
// without a tensor-core congruence.
//
// Operands are fixed point with one scale per matrix (qcs_fixed.cuh) held as packed limbs
// {re.h, re.l, im.h, im.l}, 16 bytes like an FP64 complex number.  A complex multiply-add
// takes three real products by the sums of the parts (Re = sum ur qr - sum ui qi,
// Im = sum us qs - sum ur qr - sum ui qi, formed on the limbs: two additions a factor), nine
// IMAD.WIDE or 37 clocks per 32 of them, against three DFMA or 229 clocks.  The walker's
// orbitals are in echelon form with rows of norm at most one, so their zeros are skipped and
// one scale loses nothing (the reduced form [I; X], with entries up to 16, would cost the
// others four bits).
//
// T is held in 56 bits as two limbs of 28: the dropped products of the lower limbs are below
// 2^54, a quarter of what limbs of 29 drop, and B keeps 56 bits instead of 54 (n = 6, ne = 4:
// pair errors of 4 10^-16 rms instead of 1.1 10^-15; the same instructions).
//
// Ranges, for rows of any values: a sum's hh and cr are formed modulo 2^64, so partial sums and
// the three products' own sums may wrap, but the final hh, cr and value must stay below 2^63.
// Per real product |h h'| and |h l'| + |l h'| are at most
//     T (57 bits times 57, S = 29):  2^56, 2^57    2n products: 2^61.6, 2^62.6 (n = 24)
//     B from T (56 times 56, S = 28): 2^56, 2^56   4n products: 2^62.6, 2^62.6, value 2^62.6
//     B from K (56 times 57, S = 29): 2^55, 2^55 + 2^56   4n products: 2^61.6, and for cr
//         2^62.7: a walker row has norm one, so its parts sum to at most sqrt(2n) of it, 28 of
//         48 times the scale 2^-2 that its largest part has at least (n = 24).
#pragma once
#include "qcs_fixed.cuh"

constexpr int kFxS = 29;   // the limbs of this file: X = h 2^29 + l
constexpr int kFxST = 28;  // ... of T, both factors of B: 56 bits in two equal limbs

// Bits of the local energy's Mt and K ell, of which A'_ab = sum over 2n columns of
// K_a M_b - K_b M_a, four real products each: |h l'| + |l h'| are below 2^56 at 56 bits, a cr of
// up to 8n 2^56 (2^63.6 at n = 24), so one bit less above 16 modes.
__host__ __device__ constexpr int fx_ap_bits(int n) { return n <= 16 ? 56 : 55; }

__device__ __forceinline__ fxl fx_re(int4 q) { return fxl{q.x, q.y}; }
__device__ __forceinline__ fxl fx_im(int4 q) { return fxl{q.z, q.w}; }
__device__ __forceinline__ fxl fx_add(fxl a, fxl b) { return fxl{a.h + b.h, a.l + b.l}; }
__device__ __forceinline__ fxl fx_sub(fxl a, fxl b) { return fxl{a.h - b.h, a.l - b.l}; }
__device__ __forceinline__ fxacc fx_accadd(fxacc a, fxacc b) { return fxacc{a.hh + b.hh, a.cr + b.cr}; }
__device__ __forceinline__ fxacc fx_accsub(fxacc a, fxacc b) { return fxacc{a.hh - b.hh, a.cr - b.cr}; }

// The largest upper word of |entry| of count complex FP64 numbers, over a warp.
__device__ __forceinline__ unsigned fx_max_key(const cd *__restrict__ src, int count, int lane) {
    unsigned k = 0u;
    for (int e = lane; e < count; e += 32) {
        const unsigned h = pivot_key(src[e]);
        k = h > k ? h : k;
    }
    return __reduce_max_sync(QCS_FULL, k);
}
// Whether more than one in 32, and four, of the parts that are not zero, of count complex FP64
// numbers, lie below 2^-kFxSpan of the largest (key: its upper word), over a warp: one in a
// hundred of a random walker's do, a quarter of one's at 10^-2 from a basis determinant.
constexpr int kFxSpan = 8;
__device__ __forceinline__ bool fx_wide(const cd *__restrict__ src, int count, unsigned key, int lane) {
    const int lim = (int)(key >> 20) - kFxSpan;
    unsigned small = 0u, all = 0u;
    for (int e = lane; e < count; e += 32) {
        const cd x = src[e];
        const double parts[2] = {x.x, x.y};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned nz = (__double_as_longlong(parts[h]) << 1) != 0ll;
            all += nz;
            small += nz & (unsigned)((int)(((unsigned)__double2hiint(parts[h]) >> 20) & 0x7ff) < lim);
        }
    }
    return 32u * __reduce_add_sync(QCS_FULL, small) > __reduce_add_sync(QCS_FULL, all) + 128u;
}
// Fraction bits with |x| 2^f < 2^bits for entries whose largest upper word is key.
__device__ __forceinline__ int fx_fraction(unsigned key, int bits) { return bits + 1022 - (int)(key >> 20); }

__device__ __forceinline__ int4 fx_limbs(cd x, int f) { return fx_pack(fx_split<kFxS>(fx_of1(x.x, f)), fx_split<kFxS>(fx_of1(x.y, f))); }

// count / n rows of n complex FP64 numbers (global) as limbs in padded rows of n + 1, row c
// scaled by 2^{f + rs[c]} (rs null: by 2^f).
__device__ __forceinline__ void fx_stage_rows(int n, int count, const cd *__restrict__ src, int f,
                                              const int8_t *__restrict__ rs, int4 *__restrict__ dst, int t, int nthr) {
    for (int e = t; e < count; e += nthr) {
        const int c = e / n, k = e - c * n;
        dst[c * (n + 1) + k] = fx_limbs(src[e], rs ? f + rs[c] : f);
    }
}

// Exponents that bring the two rows of each Majorana pair (2k, 2k + 1) of a snapshot's rows
// (2n x n) to the same size: B^(s) holds products of the two only, so scaling them by 2^D and
// 2^-D changes nothing, and rows of very different sizes (a Q that is not orthogonal) keep
// their precision under the one scale of T.  Returns the key of the largest balanced entry
// (at least 0x7ff00000 when an entry is not finite); every warp of a team writes the same rs.
__device__ __forceinline__ unsigned fx_balance_rows(int n, const cd *__restrict__ Q, int8_t *__restrict__ rs, int lane) {
    int most = 0;
    bool bad = false;
    for (int c0 = 0; c0 < 2 * n; c0 += 32) {
        const int c = c0 + lane;
        unsigned k = 0u;
        if (c < 2 * n)
            for (int j = 0; j < n; ++j) {
                const unsigned h = pivot_key(Q[c * n + j]);
                k = h > k ? h : k;
            }
        bad |= k >= 0x7ff00000u;
        const int e = (int)(k >> 20), o = __shfl_xor_sync(QCS_FULL, e, 1);
        int D = (c & 1) ? -((e - o) >> 1) : (o - e) >> 1;
        if (e == 0 || o == 0) D = 0;
        D = D > 100 ? 100 : D < -100 ? -100 : D;
        if (c < 2 * n) rs[c] = (int8_t)D;
        most = e != 0 && e + D > most ? e + D : most;
    }
    most = __reduce_max_sync(QCS_FULL, most);
    return __any_sync(QCS_FULL, bad) ? 0x7ff00000u : (unsigned)(most > 0 ? most : 0) << 20;
}

// Columns c0 .. c0+n-1 of T (n rows of stride ld_t, as integers worth V 2^{58-fU-fQ}) from n
// staged snapshot rows; walker row j < ne is zero in columns k < j, row ne + j' in columns
// [ne, ne + j').  Returns this thread's OR of the upper words.
__device__ inline unsigned fx_build_T(int n, int ne, const int4 *__restrict__ U, const int4 *__restrict__ Q,
                                      fx2 *__restrict__ Tv, int c0, int t, int nthr) {
    const int lu = n + 1, lt = ld_t(n);
    unsigned top = 0u;
#pragma unroll 1
    for (int e = t; e < n * n; e += nthr) {
        const int j = e / n, c = e - j * n;
        const int4 *ur = U + j * lu, *qr = Q + c * lu;
        fxacc p1 = {0, 0}, p2 = {0, 0}, p3 = {0, 0};
        int k = j < ne ? j : 0;
#pragma unroll 1
        while (k < n) {
            if (k == ne && j > ne) {  // the completion row's zeros
                k = j;
            }
            const int4 u = ur[k], q = qr[k];
            fx_mac(p1, fx_re(u), fx_re(q));
            fx_mac(p2, fx_im(u), fx_im(q));
            fx_mac(p3, fx_add(fx_re(u), fx_im(u)), fx_add(fx_re(q), fx_im(q)));
            ++k;
        }
        fxacc re = fx_accsub(p1, p2), im = fx_accsub(fx_accsub(p3, p1), p2);
        re.cr += fx_half<kFxS>(58);
        im.cr += fx_half<kFxS>(58);
        const fx2 v = make_longlong2(fx_value<kFxS>(re, 58), fx_value<kFxS>(im, 58));
        top |= fx_top(v);
        Tv[j * lt + c0 + c] = v;
    }
    return top;
}

// T of a signed-permutation snapshot: row c of Qt has one nonzero entry, the phase
// code & 3 at column code >> 2, so T[j][c] = Ut[j][k_c] ph_c is a gather, of 56 bits (worth
// V 2^{1-fU}).
__device__ inline void fx_gather_T(int n, const int4 *__restrict__ U, const uint8_t *__restrict__ code,
                                   int4 *__restrict__ T, int t, int nthr) {
    const int n2 = 2 * n, lt = ld_t(n);
    for (int e = t; e < n * n2; e += nthr) {
        const int j = e / n2, c = e - j * n2;
        const unsigned q = code[c], ph = q & 3u;
        const int4 u = U[j * (n + 1) + (int)(q >> 2)];
        const fxl a = (ph & 1u) ? fx_im(u) : fx_re(u), b = (ph & 1u) ? fx_re(u) : fx_im(u);
        long long re = (((long long)a.h << kFxS) + a.l + 1) >> 1, im = (((long long)b.h << kFxS) + b.l + 1) >> 1;
        if (ph == 1u || ph == 2u) re = -re;
        if (ph >= 2u) im = -im;
        T[j * lt + c] = fx_pack(fx_split<kFxST>(re), fx_split<kFxST>(im));
    }
}

// n x 2n integers of T in place as limbs, the largest (b bits) shifted to 56 bits.
template <int S>
__device__ __forceinline__ void fx_T_limbs(int n, void *T, int b, int t, int nthr) {
    const int n2 = 2 * n, lt = ld_t(n);
    fx2 *v = reinterpret_cast<fx2 *>(T);
    int4 *q = reinterpret_cast<int4 *>(T);
#pragma unroll 1
    for (int e = t; e < n * n2; e += nthr) {
        const int j = e / n2, i = j * lt + e - j * n2;
        const fx2 x = fx_shift(v[i], 56 - b);
        q[i] = fx_pack(fx_split<S>(x.x), fx_split<S>(x.y));
    }
}

// Real part (odd = false) or imaginary part of a limb entry.
__device__ __forceinline__ fxl fx_part(int4 q, bool odd) { return odd ? fx_im(q) : fx_re(q); }

// B^(s) (packed, the empty modes' rows first, worth X 2^{56-2f} for T worth 2^-f) from T: row c
// of an empty mode j = ne + c/2 is Re T_j (c even) or -Im T_j (c odd), the occupied row x is
// T_x; B_ab = sum_k X_a,2k X_b,2k+1 - X_a,2k+1 X_b,2k.  One loop per block (real x real, real x
// complex, complex x complex).  Returns this thread's OR of the upper words.
__device__ inline unsigned fx_build_B(int n, int ne, const int4 *__restrict__ T, fx2 *__restrict__ B,
                                      const uint16_t *__restrict__ tab, int t, int nthr) {
    const int d2 = 2 * (n - ne), lt = ld_t(n);
    unsigned top = 0u;
#pragma unroll 1
    for (int e = t; e < tri_count(d2); e += nthr) {
        int a, b;
        pair_of(tab, e, a, b);
        const bool oa = a & 1, ob = b & 1;
        const int4 *ra = T + (ne + (a >> 1)) * lt, *rb = T + (ne + (b >> 1)) * lt;
        fxacc s = {0, fx_half<kFxST>(56)};
#pragma unroll 1
        for (int k = 0; k < n; ++k) {
            fx_mac(s, fx_part(ra[2 * k], oa), fx_part(rb[2 * k + 1], ob));
            fx_mac(s, fx_neg(fx_part(ra[2 * k + 1], oa)), fx_part(rb[2 * k], ob));
        }
        const long long v = fx_value<kFxST>(s, 56);
        const fx2 x = make_longlong2(oa != ob ? -v : v, 0ll);
        top |= fx_top(x);
        B[e] = x;
    }
#pragma unroll 1
    for (int e = t; e < d2 * ne; e += nthr) {
        const int x = e / d2, c = e - x * d2;
        const bool odd = c & 1;
        const int4 *rc = T + (ne + (c >> 1)) * lt, *rx = T + x * lt;
        fxacc re = {0, fx_half<kFxST>(56)}, im = {0, fx_half<kFxST>(56)};
#pragma unroll 1
        for (int k = 0; k < n; ++k) {
            const fxl c0 = fx_part(rc[2 * k], odd), c1 = fx_neg(fx_part(rc[2 * k + 1], odd));
            const int4 x0 = rx[2 * k], x1 = rx[2 * k + 1];
            fx_mac(re, c0, fx_re(x1));
            fx_mac(im, c0, fx_im(x1));
            fx_mac(re, c1, fx_re(x0));
            fx_mac(im, c1, fx_im(x0));
        }
        const fx2 v = fx_neg_if(make_longlong2(fx_value<kFxST>(re, 56), fx_value<kFxST>(im, 56)), odd);
        top |= fx_top(v);
        B[tri_index(c, d2 + x)] = v;
    }
#pragma unroll 1
    for (int e = t; e < tri_count(ne); e += nthr) {
        int a, b;
        pair_of(tab, e, a, b);
        const int4 *ra = T + a * lt, *rb = T + b * lt;
        fxacc re = {0, fx_half<kFxST>(56)}, im = {0, fx_half<kFxST>(56)};
#pragma unroll 1
        for (int k = 0; k < n; ++k) {
            const int4 a0 = ra[2 * k], a1 = ra[2 * k + 1], b0 = rb[2 * k], b1 = rb[2 * k + 1];
            fx_mac(re, fx_re(a0), fx_re(b1));
            fx_mac(im, fx_re(a0), fx_im(b1));
            fx_mac(re, fx_neg(fx_im(a0)), fx_im(b1));
            fx_mac(im, fx_im(a0), fx_re(b1));
            fx_mac(re, fx_neg(fx_re(a1)), fx_re(b0));
            fx_mac(im, fx_neg(fx_re(a1)), fx_im(b0));
            fx_mac(re, fx_im(a1), fx_im(b0));
            fx_mac(im, fx_neg(fx_im(a1)), fx_re(b0));
        }
        const fx2 v = make_longlong2(fx_value<kFxST>(re, 56), fx_value<kFxST>(im, 56));
        top |= fx_top(v);
        B[tri_index(d2 + a, d2 + b)] = v;
    }
    return top;
}

// B^(s) (as above, worth X 2^{58-fK-fU}) from K = Ut [H1 | G2] and the walker rows: with
// W1 = K1 Ut^T = T J T^T and W2 = K2 Ut^H = T J conj(T)^T and the empty rows R_j = Re T_j,
// I_j = -Im T_j,
//     occupied a < b:             W1[a][b]
//     occupied a, empty mode j:   (a, R_j) = (W1 + W2)[a][j] / 2,  (a, I_j) = i (W1 - W2)[a][j] / 2
//     empty modes j1 <= j2 (al = W1, be = W2 at [j1][j2]):
//         (R, R) = Re(al + be)/2, (R, I) = Im(be - al)/2, (I, R) = -Im(al + be)/2,
//         (I, I) = Re(be - al)/2; within one mode only (R_j, I_j) = Im(be)/2.
// n-term sums over the non-zero columns of walker row b instead of the 2n of T: above 16
// modes cheaper than fx_build_B.  Three real products per complex term:
//     K1 u:       Re = p1 - p2, Im = p3 - p1 - p2,   p3 = sum (k1r + k1i)(ur + ui)
//     K2 conj(u): Re = q1 + q2, Im = q1 - q2 - q3,   q3 = sum (k2r - k2i)(ur + ui)
// The occupied-empty and empty-empty items share their sums' shape, so they run in one loop
// ordered by completion row b: neighbouring lanes share their loop bounds.
__device__ inline unsigned fx_build_B_from_K(int n, int ne, const int4 *__restrict__ U, const int4 *__restrict__ K,
                                             fx2 *__restrict__ B, const uint16_t *__restrict__ tab, int t, int nthr) {
    const int d = n - ne, d2 = 2 * d, lu = n + 1, lt = ld_t(n);
    unsigned top = 0u;
    auto put = [&](int i, int j, fx2 v) {  // i < j
        top |= fx_top(v);
        B[tri_index(i, j)] = v;
    };
    auto whole = [](fxacc s) {
        s.cr += fx_half<kFxS>(58);
        return fx_value<kFxS>(s, 58);
    };
    auto half = [&](fxacc s) { return (whole(s) + 1) >> 1; };
#pragma unroll 1
    for (int e = t; e < tri_count(ne); e += nthr) {
        int a, b;
        pair_of(tab, e, a, b);
        const int4 *kr = K + a * lt, *ur = U + b * lu;
        fxacc p1 = {0, 0}, p2 = {0, 0}, p3 = {0, 0};
#pragma unroll 1
        for (int k = b; k < n; ++k) {
            const int4 kk = kr[k], u = ur[k];
            fx_mac(p1, fx_re(kk), fx_re(u));
            fx_mac(p2, fx_im(kk), fx_im(u));
            fx_mac(p3, fx_add(fx_re(kk), fx_im(kk)), fx_add(fx_re(u), fx_im(u)));
        }
        put(d2 + a, d2 + b,
            make_longlong2(whole(fx_accsub(p1, p2)), whole(fx_accsub(fx_accsub(p3, p1), p2))));
    }
    const int c2 = ne * d + tri_count(d + 1);
    int jj = 0, base = 0;  // completion row b = ne + jj carries ne + jj + 1 items
#pragma unroll 1
    for (int e = t; e < c2; e += nthr) {
        while (jj + 1 < d && base + ne + jj + 1 <= e) {
            base += ne + jj + 1;
            ++jj;
        }
        const int i = e - base, b = ne + jj;  // K row i: an occupied row, or that of empty mode i - ne
        const int4 *kr = K + i * lt, *ur = U + b * lu;
        fxacc p1 = {0, 0}, p2 = {0, 0}, p3 = {0, 0}, q1 = {0, 0}, q2 = {0, 0}, q3 = {0, 0};
        int k = 0;
#pragma unroll 1
        while (k < n) {
            if (k == ne && b > ne) k = b;
            const int4 u = ur[k], k1 = kr[k], k2 = kr[n + k];
            const fxl ur_ = fx_re(u), ui_ = fx_im(u), us = fx_add(ur_, ui_);
            fx_mac(p1, fx_re(k1), ur_);
            fx_mac(p2, fx_im(k1), ui_);
            fx_mac(p3, fx_add(fx_re(k1), fx_im(k1)), us);
            fx_mac(q1, fx_re(k2), ur_);
            fx_mac(q2, fx_im(k2), ui_);
            fx_mac(q3, fx_sub(fx_re(k2), fx_im(k2)), us);
            ++k;
        }
        const fxacc w1x = fx_accsub(p1, p2), w1y = fx_accsub(fx_accsub(p3, p1), p2);
        const fxacc w2x = fx_accadd(q1, q2), w2y = fx_accsub(fx_accsub(q1, q2), q3);
        const long long xs = half(fx_accadd(w1x, w2x)), ys = half(fx_accadd(w1y, w2y));
        const long long xd = half(fx_accsub(w1x, w2x)), yd = half(fx_accsub(w1y, w2y));
        if (i < ne) {  // (empty, occupied) entries: the negatives
            put(2 * jj, d2 + i, make_longlong2(-xs, -ys));
            put(2 * jj + 1, d2 + i, make_longlong2(yd, -xd));
        } else {
            const int r1 = 2 * (i - ne), r2 = 2 * jj;
            if (r1 < r2) {
                put(r1, r2, make_longlong2(xs, 0));
                put(r1, r2 + 1, make_longlong2(-yd, 0));
                put(r1 + 1, r2, make_longlong2(-ys, 0));
                put(r1 + 1, r2 + 1, make_longlong2(-xd, 0));
            } else {
                put(r1, r1 + 1, make_longlong2(half(w2y), 0));
            }
        }
    }
    return top;
}
