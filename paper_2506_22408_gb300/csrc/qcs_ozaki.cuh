// qcs_ozaki.cuh -- error-free slicing of FP64 operands for tensor-core products.
//
// A real row x (FP64) with row scale 2^e (max |x_k| (1 + 2^-7) < 2^e) is written as
//     x_k = 2^{e-55} u_k,  u_k = sum_{i=1..7} a_ik 2^{8(7-i)},  a_ik integers in [-128, 127],
// i.e. x_k 2^{55-e} rounded to an integer |u_k| < 2^55 - 2^47 in balanced base 256: the
// bytes of u_k + 0x80808080808080, each less 128.  Every slice is exact in BF16.  The
// product of two sliced rows is
//     sum_k x_k y_k = 2^{e+f+2} sum_{L=2..14} 2^{-8L} sum_{i+j=L} sum_k a_ik b_jk,
// and each level sum sum_{i+j=L} sum_k a_ik b_jk is an integer of magnitude at most
// 7 * 32 * 128^2 < 2^22 for K = 32 terms and at most 7 products per level, so the
// tensor cores accumulate it exactly in FP32 (no rounding anywhere), and one FP32 addition
// of 1.5 2^23 leaves it in the low bits of the sum's pattern.  Levels L = 2..8 are formed;
// the dropped ones (L >= 9, digits of either sign) and the rounding of the slices bound the
// error by about 2^-53 of sum_k |x_k||y_k| relative to the row scales, the size of the
// rounding error of an FP64 dot product of the same length (Ozaki, Ogita, Oishi and Rump's
// error-free splitting of matrix products, with integer-valued slices).
//
// Balanced digits need no sign beside them: slicing an entry takes one 64-bit addition and
// per digit a byte permutation, an FP32 addition and half a pack, and no level sum takes a
// float-to-integer conversion (sign-magnitude slices: 35 % of that unit's cycles; 1024 x
// 20000 overlaps at n = 16 took 250.1 ms with them, 248.8 without).  The levels keep two bits
// below the last level's carry, as much as fits 64 bits.
//
// The levels are combined exactly in integer arithmetic into one 64-bit fixed-point value
// z = sum_{L=2..7} acc_L 2^{8(7-L)+2} + floor(acc_8 / 2^6 + 1/2), worth z 2^{e+f-56}; |z| < 2^62.
// Nothing in this file issues an FP64 instruction except fixed_to_f64_exact, the path for
// exponents outside the normal range.
#pragma once
#include <stdint.h>

#include "qcs_common.cuh"

namespace qcs_oz {

constexpr int kSlices = 7;             // 8-bit slices per operand: 56 bits
constexpr int kLevels = kSlices;       // product levels L = 2..8 that are formed
constexpr int kRowsPer = 32;           // padded rows / contraction length of one operand (2n <= 32)
constexpr int kSliceBytes = kRowsPer * kRowsPer * 2;  // one 32 x 32 BF16 slice (K-major core matrices)
constexpr int kNoRow = -100000;        // row scale of an all-zero row

// Byte offset of element (row, k) of a 16-bit K-major operand with 32 columns and no
// swizzle: 8-row x 16-byte core matrices, K-adjacent ones 128 bytes apart (LBO),
// row-adjacent groups of 8 rows 512 bytes apart (SBO).
__host__ __device__ __forceinline__ uint32_t kmajor16(int row, int k) {
    return (uint32_t)((row >> 3) * 512 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

constexpr uint64_t kDigitBias = 0x80808080808080ull;

// Digit i (1..7) of u = sum a_i 2^{8(7-i)} from b = u + kDigitBias, as an FP32: byte 7 - i of
// b is placed under the exponent of 2^23 (bit pattern 0x4B0000bb, the value 2^23 + byte) by
// one byte permutation; less 2^23 + 128 it is exact.  With i a compile-time constant the
// word and byte selection fold away.
__device__ __forceinline__ float slice_f32(uint64_t b, int i) {
    const int byte = 7 - i;
    const uint32_t w = byte >= 4 ? (uint32_t)(b >> 32) : (uint32_t)b;
    return __uint_as_float(__byte_perm(w, 0x4B000000u, (uint32_t)(byte & 3) | 0x7440u)) - 8388736.0f;
}

// Two FP32 values that BF16 holds exactly (integers of magnitude <= 255) as one BF16
// pair, lo first in memory (the lower half of the word).
__device__ __forceinline__ uint32_t bf16x2_of(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Exponent e with |x| (1 + 2^-7) < 2^e for a finite nonzero x, from the bit pattern (no FP64
// instruction).  Subnormals are treated as 2^-1022.
__device__ __forceinline__ int row_exp_of(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    const int hx = (int)((b + (1ull << 46)) >> 52);  // a carry out of the mantissa above 1 - 2^-7 of 2
    return (hx == 0 ? 1 : hx) - 1023 + 1;
}

// x 2^{55-e} rounded to an integer (|x| (1 + 2^-7) < 2^e), from the bit pattern.
__device__ __forceinline__ long long fixed_of(double x, int e) {
    const long long b = __double_as_longlong(x);
    const int hx = (int)((b >> 52) & 0x7ff);
    if (hx == 0) return 0ll;  // zeros (and subnormals, far below any row scale here)
    const long long m = (b & ((1ll << 52) - 1)) | (1ll << 52);  // |x| = m 2^{hx-1075}
    const int sh = hx - 1075 + 55 - e;                             // |u| = m 2^sh, sh <= 2
    const int r = sh < 0 ? (sh > -62 ? -sh : 62) : 0;              // m < 2^53: zero from 55 on
    const long long u = ((m << (sh > 0 ? (sh < 2 ? sh : 2) : 0)) + ((1ll << r) >> 1)) >> r;
    return b < 0 ? -u : u;
}

// z = sum_{L=2..7} acc[L-2] 2^{8(7-L)+2} + floor(acc[6] / 2^6 + 1/2) for the seven level sums
// acc[0..6] (levels 2..8) of one output entry, integers of magnitude below 2^22: acc + 1.5 2^23
// has the bit pattern kMagic + acc, and the patterns' multiples of kMagic are taken off
// together.  Levels 2 and 3 only touch the upper word.
__device__ __forceinline__ long long combine_levels(const float (&acc)[kLevels]) {
    constexpr unsigned kMagic = 0x4B400000u;
    constexpr unsigned long long kOff =
        (unsigned long long)kMagic * 0x0000040404040404ull + (unsigned long long)(kMagic >> 6);
    unsigned x[kLevels];
#pragma unroll
    for (int L = 0; L < kLevels; ++L) x[L] = __float_as_uint(acc[L] + (L == kLevels - 1 ? 12582944.0f : 12582912.0f));
    unsigned long long z = (unsigned long long)x[5] * 4u + (x[6] >> 6);
    z += (unsigned long long)x[4] * 1024u;
    z += (unsigned long long)x[3] * 262144u;
    z += (unsigned long long)x[2] * 67108864u;
    z += (unsigned long long)(x[0] * 1024u + x[1] * 4u) << 32;
    return (long long)(z - kOff);
}

// Exponent G with |z| 2^g (1 + 2^-7) < 2^G, from the upper word where it is not zero (at most
// two bits above the least one), g + 33 below it; kNoRow for z = 0.  A maximum of these over
// entries of different g is a scale of them all: an entry of a zero upper word counts too, as
// its g may exceed the others'.
__device__ __forceinline__ int scale_of_fixed(long long z, int g) {
    const int zh = (int)(z >> 32), zm = zh < 0 ? -zh : zh;
    return zm != 0 ? g + 64 - __clz(zm + (zm >> 6) + 1) : z != 0 ? g + 33 : kNoRow;
}

// z 2^E as an FP64 (round to nearest on the 11 dropped bits), assembled from the bits
// with selects only, so that a warp converts its entries without diverging.  The
// exponent of the result must lie in the normal range; range_ok is cleared otherwise
// (zero is always in range), and the caller then takes fixed_to_f64_exact.
__device__ __forceinline__ double fixed_to_f64(long long z, int E, bool &range_ok) {
    const unsigned long long sg = z < 0 ? (1ull << 63) : 0ull;
    const unsigned long long u = z < 0 ? (unsigned long long)(-z) : (unsigned long long)z;
    const int lz = __clzll((long long)u);               // 64 for z = 0
    const unsigned long long nrm = u << (lz & 63);      // top bit set (0 for z = 0)
    // 53 significant bits, rounded on the first dropped bit.  Added to the exponent
    // field (ex + 1022), the leading bit 2^52 of mant raises it to ex + 1023; after a
    // rounding carry mant is 2^53, which gives ex + 1024 with a zero fraction: 2^(ex+1).
    const unsigned long long mant = (nrm >> 11) + ((nrm >> 10) & 1ull);
    const int ex = 63 - lz + E;
    range_ok = range_ok && (u == 0ull || (ex >= -1020 && ex <= 1020));
    const long long bits = (long long)(sg | (((unsigned long long)(ex + 1022) << 52) + mant));
    return u == 0ull ? 0.0 : __longlong_as_double(bits);
}

// The same value for any exponent (subnormal, overflow), by ldexp.
__device__ __forceinline__ double fixed_to_f64_exact(long long z, int E) { return ldexp((double)z, E); }

// Write the seven slices of a 32-entry row (u[k] as fixed_of gives them) into the K-major
// slice slabs: slab i (1..7) starts at base + (i-1) * slab_stride bytes, the row is `row` of
// its operand.  Four 16-byte stores per slice.
__device__ __forceinline__ void store_row_slices(unsigned char *base, uint32_t slab_stride, int row,
                                                 const long long (&u)[kRowsPer]) {
#pragma unroll
    for (int i = 1; i <= kSlices; ++i) {
        unsigned char *slab = base + (size_t)(i - 1) * slab_stride;
#pragma unroll
        for (int kb = 0; kb < 4; ++kb) {
            uint4 w;
            uint32_t *wp = reinterpret_cast<uint32_t *>(&w);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int k = 8 * kb + 2 * t;
                wp[t] = bf16x2_of(slice_f32((uint64_t)u[k] + kDigitBias, i), slice_f32((uint64_t)u[k + 1] + kDigitBias, i));
            }
            *reinterpret_cast<uint4 *>(slab + kmajor16(row, 8 * kb)) = w;
        }
    }
}

}  // namespace qcs_oz
