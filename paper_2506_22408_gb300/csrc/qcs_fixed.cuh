// qcs_fixed.cuh -- the Pfaffian eliminations in 64-bit fixed point on the integer pipe.
//
// GB300 issues one 32-lane FP64 FMA per 76 clocks and SM sub-partition, but one 32 x 32 ->
// 64-bit integer multiply-add (IMAD.WIDE) per 4.1 (register-only probes).  A matrix whose
// entries share one power-of-two scale needs no exponent per entry, so the eliminations
// hold every entry as a 64-bit integer X worth X 2^-f, f common to the matrix.  A product
// of two of them takes three IMAD.WIDE on their 31-bit limbs,
//     X = h 2^31 + l,  |l| <= 2^30:   X Y = hh 2^62 + (h l' + l h') 2^31 + l l',
// the last term (below 2^-60 of the factors' scale, either sign) dropped: 12 to 13 clocks
// against 76.  The largest entry of a matrix is kept at 54 to 60 bits, so an update rounds
// at 2^-54 to 2^-60 of the matrix's largest entry where FP64 rounds at 2^-53 of each
// operand: the elimination with pivoting is as accurate as that matrix norm allows either
// way, and the errors against 64-bit references are those of the FP64 code it replaced or
// smaller.
//
// One rank-2 entry update (two complex products) is 24 IMAD.WIDE and about 35 one-clock
// instructions, near 140 clocks per 32 entries, against 8 DFMA = 611 clocks.  With the
// products that cheap, everything around them counts: matrices are ordered with the empty
// modes first and eliminated from the last index up, so that the remaining matrix is a
// prefix of the packed triangle, updated in place without index lists; pivots are compared
// on upper words; products of pivots are taken in normalised fixed point as well.
#pragma once
#include "qcs_ozaki.cuh"
#include "qcs_pair.cuh"

typedef longlong2 fx2;  // complex fixed point, worth (x + i y) 2^-f

// Bits of the largest entry: after a (re)normalisation; before an update at most (limbs of
// 31 bits) and at least.  |g| <= sqrt 2 2^eu and |v| <= sqrt 2 2^mb bound an update by
// 4 2^{mb+eu}: its result is scaled down by q bits when mb + eu exceeds kFxRoom, so that
// it stays below 2^62.4; the scale of the factors themselves is kept, which matters when
// a pivot is small (scaling the matrix down before the update would cost eu bits of g v).
constexpr int kFxTop = 58;
constexpr int kFxMax = 61;
constexpr int kFxLow = 54;
constexpr int kFxRoom = 60;

// The threads that share one pair: a warp, or two warps with a named barrier and two
// pairs of shared words for the reductions across them.
template <int NW>
struct FxTeam {
    static constexpr int NT = 32 * NW;
    static constexpr int kWarps = NW;
    int t, lane, wid, bar;
    unsigned *scr;
    __device__ __forceinline__ void sync() const {
        if (NW == 1) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(NT) : "memory");
    }
    // the OR over the team of v: every thread calls or_put, a sync() follows, then or_get
    // with the same parity bit (alternated by the caller from one reduction to the next)
    __device__ __forceinline__ unsigned or_put(unsigned v, int par) const {
        v = __reduce_or_sync(QCS_FULL, v);
        if (NW > 1 && lane == 0) scr[2 * par + wid] = v;
        return v;
    }
    __device__ __forceinline__ unsigned or_get(unsigned v, int par) const {
        return NW > 1 ? scr[2 * par] | scr[2 * par + 1] : v;
    }
};
typedef FxTeam<1> FxWarp;

struct fxl {  // a fixed-point number as limbs h 2^31 + l
    int h, l;
};
__device__ __forceinline__ fxl fx_split(long long X) {
    const int h = (int)((X + (1ll << 30)) >> 31);
    return fxl{h, (int)((unsigned)X - ((unsigned)h << 31))};
}
__device__ __forceinline__ fxl fx_neg(fxl a) { return fxl{-a.h, -a.l}; }

struct fxacc {  // hh 2^62 + cr 2^31
    long long hh, cr;
};
__device__ __forceinline__ void fx_mac(fxacc &s, fxl a, fxl b) {
    s.hh += (long long)a.h * b.h;
    s.cr += (long long)a.h * b.l;
    s.cr += (long long)a.l * b.h;
}
// (hh 2^62 + cr 2^31) 2^{-62 + up}, 0 <= up < 31
__device__ __forceinline__ long long fx_value(const fxacc &s, int up) { return (s.hh << up) + (s.cr >> (31 - up)); }

__device__ __forceinline__ int4 fx_pack(fxl re, fxl im) { return make_int4(re.h, re.l, im.h, im.l); }

// Bits of max(|re|, |im|) (0 for a zero entry).
__device__ __forceinline__ unsigned long long fx_mag(fx2 a) {
    const unsigned long long x = (unsigned long long)(a.x < 0 ? -a.x : a.x), y = (unsigned long long)(a.y < 0 ? -a.y : a.y);
    return x > y ? x : y;
}
__device__ __forceinline__ int fx_bits(fx2 a) { return 64 - __clzll((long long)fx_mag(a)); }

// Pivot key of 26 bits: the bit length of max(|re|, |im|), then its next 19 bits, so that
// keys order like magnitudes to a relative 2^-19; 0 for a zero entry only.
__device__ __forceinline__ unsigned fx_key(fx2 a) {
    const unsigned long long m = fx_mag(a);
    if (m == 0ull) return 0u;
    const int lz = __clzll((long long)m);
    return ((unsigned)(64 - lz) << 19) + ((unsigned)((m << lz) >> 44) & 0x7ffffu);
}

// max(|re|, |im|) from the upper words (below 2^30, in units of 2^32).
__device__ __forceinline__ unsigned fx_mag32(fx2 a) {
    const int x = abs((int)(a.x >> 32)), y = abs((int)(a.y >> 32));
    return (unsigned)(x > y ? x : y);
}

// OR of the upper words of |re| and |im|: over any set of entries, the top bit of the OR is
// that of the largest magnitude.
__device__ __forceinline__ unsigned fx_top(fx2 a) {
    return (unsigned)abs((int)(a.x >> 32)) | (unsigned)abs((int)(a.y >> 32));
}
__device__ __forceinline__ int fx_top_bits(unsigned top) { return 64 - __clz((int)top); }  // 32 if top == 0

// X 2^s, rounded to nearest when s < 0.
__device__ __forceinline__ long long fx_shift1(long long X, int s) {
    if (s >= 0) return X << (s < 63 ? s : 63);
    return s < -62 ? 0ll : (X + (1ll << (-s - 1))) >> (-s);
}
__device__ __forceinline__ fx2 fx_shift(fx2 a, int s) { return make_longlong2(fx_shift1(a.x, s), fx_shift1(a.y, s)); }

// The same without a branch.
__device__ __forceinline__ long long fx_shift_any(long long X, int s) {
    const int r = s < 0 ? (s > -63 ? -s : 63) : 0;
    const long long y = X << (s > 0 ? s : 0);
    return (y + ((1ll << r) >> 1)) >> r;
}

// x 2^f rounded to an integer, from the bit pattern (|x| 2^f < 2^62; no FP64 instruction).
__device__ __forceinline__ long long fx_of1(double x, int f) {
    const long long b = __double_as_longlong(x);
    const int hx = (int)((b >> 52) & 0x7ff);
    const long long m = (b & ((1ll << 52) - 1)) | (hx ? (1ll << 52) : 0ll);
    const long long u = fx_shift1(m, (hx ? hx : 1) - 1075 + f);
    return b < 0 ? -u : u;
}
__device__ __forceinline__ fx2 fx_of(cd x, int f) { return make_longlong2(fx_of1(x.x, f), fx_of1(x.y, f)); }

// X 2^E as an FP64.
__device__ __forceinline__ double fx_f64(long long X, int E) {
    bool ok = true;
    const double v = qcs_oz::fixed_to_f64(X, E, ok);
    return ok ? v : qcs_oz::fixed_to_f64_exact(X, E);
}

// Entry (i, j), i != j, of a packed skew-symmetric matrix.
__device__ __forceinline__ fx2 fx_skew(const fx2 *__restrict__ N, int i, int j) {
    const bool lo = i > j;
    const fx2 v = N[lo ? tri_index(j, i) : tri_index(i, j)];
    const long long m = lo ? -1ll : 0ll;
    return make_longlong2((v.x ^ m) - m, (v.y ^ m) - m);
}

// A(i, j) = x, A(j, i) = -x.
__device__ __forceinline__ void fx_put(fx2 *__restrict__ N, int i, int j, fx2 x) {
    const long long m = i > j ? -1ll : 0ll;
    N[i > j ? tri_index(j, i) : tri_index(i, j)] = make_longlong2((x.x ^ m) - m, (x.y ^ m) - m);
}

// 1 / (q.x + i q.y) 2^119 as limbs, for max(|q.x|, |q.y|) in [2^60, 2^61): conj(q) / |q|^2,
// the reciprocal R = 2^118 / (|q|^2 2^-62) by one third-order step from the FP32 seed R0
// (relative error e < 2^-22: R = R0 (1 + e + e^2), e^3 < 2^-66) in integers.
__device__ __forceinline__ void fx_inverse(fx2 q, fxl &ir, fxl &ii) {
    const fxl a = fx_split(q.x), b = fx_split(q.y);
    fxacc s = {0, 0};
    fx_mac(s, a, a);
    fx_mac(s, b, b);
    const long long D = s.hh + (s.cr >> 31);  // |q|^2 2^-62 in [2^58, 2^61]
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"((float)(int)(D >> 31)));
    const int R0 = (int)(y * 18014398509481984.0f);  // 2^54 y in [2^24, 2^27]
    const long long e = -(long long)((unsigned long long)D * (unsigned long long)(long long)R0);  // 2^85 (1 - D R0 2^-85)
    const int eh = (int)(e >> 32);
    const int e2 = __mulhi(eh, eh);
    const long long R = ((long long)R0 << 33) + (((long long)R0 * eh) >> 20) +
                        (long long)(((unsigned long long)(unsigned)R0 * (unsigned)e) >> 52) + (((long long)R0 * e2) >> 41);
    const fxl r = fx_split(R);
    fxacc u = {0, 0}, v = {0, 0};
    fx_mac(u, a, r);
    fx_mac(v, b, r);
    ir = fx_split(fx_value(u, 1));
    ii = fx_neg(fx_split(fx_value(v, 1)));
}

// z I 2^-60 for I = 2^119 / q as limbs: 2^59 z / q, as packed limbs.
__device__ __forceinline__ int4 fx_times_inverse(fx2 z, fxl ir, fxl ii) {
    const fxl a = fx_split(z.x), b = fx_split(z.y);
    fxacc re = {0, 0}, im = {0, 0};
    fx_mac(re, a, ir);
    fx_mac(re, b, fx_neg(ii));
    fx_mac(im, a, ii);
    fx_mac(im, b, ir);
    return fx_pack(fx_split(fx_value(re, 2)), fx_split(fx_value(im, 2)));
}

// A complex number (x + i y) 2^e, the larger part of 60 bits unless it is zero.
struct fxp {
    long long x, y;
    int e;
};
__device__ __forceinline__ fxp fx_norm(fx2 a, int e) {
    const int sh = 60 - fx_bits(a);
    const fx2 z = fx_shift(a, sh < 60 ? sh : 0);
    return fxp{z.x, z.y, e - sh};
}
__device__ __forceinline__ fxp fx_prod(const fxp &a, const fxp &b) {
    const fxl ar = fx_split(a.x), ai = fx_split(a.y), br = fx_split(b.x), bi = fx_split(b.y);
    fxacc re = {0, 0}, im = {0, 0};
    fx_mac(re, ar, br);
    fx_mac(re, fx_neg(ai), bi);
    fx_mac(im, ar, bi);
    fx_mac(im, ai, br);
    return fx_norm(make_longlong2(fx_value(re, 0), fx_value(im, 0)), a.e + b.e + 62);
}
__device__ __forceinline__ fxp fx_shfl_xor(const fxp &a, int o) {
    return fxp{__shfl_xor_sync(QCS_FULL, a.x, o), __shfl_xor_sync(QCS_FULL, a.y, o), __shfl_xor_sync(QCS_FULL, a.e, o)};
}

// Rank-2 update, in place, of the leading rv x rv blocks of nb packed matrices (stride T):
//     A_ij = (A_ij + g_i v_j - v_i g_j) 2^-q,   g scaled by 2^{59-eu}.
// Entry t of the packed triangle is read and written by one thread; (i, j) comes from the
// pair table.  Returns this thread's OR of the new entries' upper words.
template <class Team>
__device__ __forceinline__ unsigned fx_rank2(const Team &tm, int nb, int T, int rv, fx2 *__restrict__ Ns,
                                             const int4 *__restrict__ Gv, const int4 *__restrict__ Vv, int ldv, int eu,
                                             int q, const uint16_t *__restrict__ tab) {
    const int Tr = tri_count(rv), total = nb * Tr;
    const int up = 3 + eu - q;
    unsigned top = 0u;
    int u = tm.t;
    const int4 *G = Gv, *V = Vv;
    fx2 *N = Ns;
    for (int e = tm.t; e < total; e += Team::NT) {
        while (u >= Tr) {
            u -= Tr;
            N += T;
            G += ldv;
            V += ldv;
        }
        int ia, ib;
        pair_of(tab, u, ia, ib);
        fx2 x = N[u];
        const int4 gi = G[ia], vi = V[ia], gj = G[ib], vj = V[ib];
        const fxl gir = {gi.x, gi.y}, gii = {gi.z, gi.w}, gjr = {gj.x, gj.y}, gji = {gj.z, gj.w};
        const fxl vir = {vi.x, vi.y}, vii = {vi.z, vi.w}, vjr = {vj.x, vj.y}, vji = {vj.z, vj.w};
        const fxl mgii = fx_neg(gii), mvir = fx_neg(vir), mvii = fx_neg(vii);
        fxacc re = {0, 0}, im = {0, 0};
        fx_mac(re, gir, vjr);
        fx_mac(im, gir, vji);
        fx_mac(re, mgii, vji);
        fx_mac(im, gii, vjr);
        fx_mac(re, mvir, gjr);
        fx_mac(im, mvir, gji);
        fx_mac(re, vii, gji);
        fx_mac(im, mvii, gjr);
        if (q > 0) {
            x.x >>= q;
            x.y >>= q;
        }
        x.x += fx_value(re, up);
        x.y += fx_value(im, up);
        top |= fx_top(x);
        N[u] = x;
        u += Team::NT;
    }
    return top;
}

// Multiply the entries of nb packed matrices (tri(r) entries each, stride T) by 2^sh.
template <class Team>
__device__ __noinline__ void fx_renorm(const Team &tm, int nb, int T, int r, fx2 *Ns, int sh) {
    const int Tr = tri_count(r);
    tm.sync();
    for (int w = 0; w < nb; ++w)
        for (int u = tm.t; u < Tr; u += Team::NT) Ns[w * T + u] = fx_shift(Ns[w * T + u], sh);
    tm.sync();
}

// Records of fx_node_pfaffians' products per warp for NB node matrices per round (vm: the
// entries of the kernel's Gauss-vector buffers, the full matrix or NB complements); the
// ne/2 signed pivots of the shared occupied elimination follow them.  A record is an entry
// worth X 2^-f with its f: 16 + 4 bytes, the f after all the entries.
__host__ __device__ inline int pv_records(int vm, int NB) { return vm / 2 + NB; }
__host__ __device__ inline size_t pv_bytes(int vm, int NB, int ne) {
    return (size_t)(pv_records(vm, NB) + ne / 2) * (sizeof(fx2) + sizeof(int));
}

// Workspace of one pair in the team's shared memory, besides its matrices.
struct FxWork {
    int4 *Gv, *Vv;  // Gauss vectors as limbs: max(m, NB 2d) entries each
    fx2 *pv;        // records
    int *pe;        // ... and their fraction bits
    int npv;        // index of the first occupied pivot's record
};

// Position of selected row x (occupied rows 0 .. ne-1, then the empty modes' rows) in the
// order the eliminations use: the empty modes' rows first.  ne and 2d are even, so the
// reordering keeps the Pfaffian.
__device__ __forceinline__ int fx_row(int x, int m, int ne) { return x < ne ? m - ne + x : x - ne; }

// B^(s) from its packed FP64 form in the order of the selection (Bs), as fixed point in
// the eliminations' order (Xs), the largest entry of kFxTop bits, f the fraction bits.
// Returns false when an entry is not finite.
template <class Team>
__device__ inline bool fx_load(const Team &tm, int m, int ne, const cd *__restrict__ Bs, fx2 *__restrict__ Xs, int &f,
                               const uint16_t *__restrict__ tab) {
    const int T = tri_count(m);
    unsigned kb = 0u;
    for (int e = tm.lane; e < T; e += 32) {  // every warp of the team takes the maximum itself
        const unsigned k = pivot_key(Bs[e]);
        kb = k > kb ? k : kb;
    }
    kb = __reduce_max_sync(QCS_FULL, kb);
    const int hx = (int)(kb >> 20);  // |x| < 2^{hx - 1022}
    f = kFxTop + 1022 - hx;
    if (hx == 0x7ff) return false;
    for (int e = tm.t; e < T; e += Team::NT) {
        int a, b;
        pair_of(tab, e, a, b);
        const int i = fx_row(a, m, ne), j = fx_row(b, m, ne);
        const fx2 x = fx_of(flip_if(Bs[e], i > j), f);
        Xs[i < j ? tri_index(i, j) : tri_index(j, i)] = x;
    }
    tm.sync();
    return true;
}

// Elimination of the occupied block, shared by every node matrix.  The node matrices
// B + w D differ only in their empty x empty block (D pairs the empty modes), so
// eliminating the ne occupied indices first is the same for all of them:
// pf(B + w D) = pf0 pf(S + w D_ee), S the Schur complement of the occupied block.
// In place on X (tri(m) entries, worth X 2^-f, the largest of at most mb bits).  Each step
// takes the largest entry (p, k) of the active occupied block as pivot, moves k to the
// last and p to the last but one position (a swap flips the sign) and updates the leading
// block; the ne/2 signed pivots become the records pvo (their product pf0 enters each
// node's product).  On success the leading tri(2d) entries of X hold S and f and mb are
// S's.  Returns false when a pivot is zero, an element of a Gauss vector exceeds 2^20 or
// the largest entry of S exceeds 2^8 times the largest entry of B (the caller then
// eliminates each node matrix in full).
template <class Team>
__device__ inline bool fx_schur_occupied(const Team &tm, int m, int ne, fx2 *__restrict__ X, int4 *__restrict__ Gv,
                                         int4 *__restrict__ Vv, const uint16_t *__restrict__ tab,
                                         fx2 *__restrict__ pvo, int *__restrict__ peo, int &f, int &mb) {
    const int d2 = m - ne;
    const int bound = mb - f + 8;
    for (int s = 0, r = m; r > d2; ++s, r -= 2) {
        const int ro = r - d2;  // the active occupied indices are 2d .. r - 1
        if (mb > kFxMax || mb < kFxLow) {
            fx_renorm(tm, 1, 0, r, X, kFxTop - mb);
            f += kFxTop - mb;
            mb = kFxTop;
        }
        // the largest entry of the active occupied block (every warp finds it by itself)
        unsigned bk = 0u;
        for (int t = tm.lane; t < tri_count(ro); t += 32) {
            int a, b;
            pair_of(tab, t, a, b);
            const unsigned c = ((fx_mag32(X[tri_index(d2 + a, d2 + b)]) >> 6) << 9) | (unsigned)(511 - t);
            bk = c > bk ? c : bk;
        }
        bk = __reduce_max_sync(QCS_FULL, bk);
        int bt = 511 - (int)(bk & 511u);
        if ((bk >> 9) < 64u) {  // small against the matrix: compare by the whole words
            unsigned kk = 0u, kt = 0u;
            for (int t = tm.lane; t < tri_count(ro); t += 32) {
                int a, b;
                pair_of(tab, t, a, b);
                const unsigned key = fx_key(X[tri_index(d2 + a, d2 + b)]);
                if (key > kk) {
                    kk = key;
                    kt = (unsigned)t;
                }
            }
            const unsigned top = __reduce_max_sync(QCS_FULL, kk);
            if (top == 0u) return false;  // the active occupied block is zero
            bt = (int)__reduce_min_sync(QCS_FULL, kk == top ? kt : 0xffffffffu);
        }
        int P, K;
        pair_of(tab, bt, P, K);
        P += d2;
        K += d2;
        // row K can hold larger entries than the pivot among the empty indices
        unsigned rt = 0u;
        for (int a = tm.lane; a < r; a += 32)
            if (a != K) rt |= fx_top(X[a < K ? tri_index(a, K) : tri_index(K, a)]);
        rt = __reduce_or_sync(QCS_FULL, rt);
        const fx2 piv = X[tri_index(P, K)];
        const int pb = fx_bits(piv), rb = fx_top_bits(rt);
        const int eu = rb >= pb ? rb - pb + 1 : 0;  // |g| 2^-eu < sqrt 2
        if (eu > 20) return false;
        if (tm.t == 0) {
            const bool neg = (K != r - 1) != (P != r - 2);
            pvo[s] = neg ? make_longlong2(-piv.x, -piv.y) : piv;
            peo[s] = f;
        }
        if (r == 2) break;  // no empty modes: the last pivot closes the Pfaffian
        const int sn = 61 - pb;
        fxl ir, ii;
        fx_inverse(make_longlong2(piv.x << sn, piv.y << sn), ir, ii);
        const int sP = K == r - 2 ? r - 1 : r - 2;  // what takes place P (if P stays), and r - 1 takes K
        tm.sync();  // every warp has read the pivot and row K
        const int rv = r - 2;
        for (int i = tm.t; i < rv; i += Team::NT) {
            const int o = i == K ? r - 1 : i == P ? sP : i;
            // g = A_{i,k} / A_{p,k}, v = A_{i,p}
            Gv[i] = fx_times_inverse(fx_shift(fx_skew(X, o, K), sn - eu), ir, ii);
            const fx2 v = fx_skew(X, o, P);
            Vv[i] = fx_pack(fx_split(v.x), fx_split(v.y));
            if (i != P && i != K) {
                if (K < rv) fx_put(X, i, K, fx_skew(X, i, r - 1));
                if (P < rv) fx_put(X, i, P, fx_skew(X, i, sP));
            } else if (i == K && P < rv) {
                fx_put(X, P, K, fx_skew(X, sP, r - 1));
            }
        }
        tm.sync();
        const int q = mb + eu > kFxRoom ? mb + eu - kFxRoom : 0;
        unsigned o = fx_rank2(tm, 1, 0, rv, X, Gv, Vv, 0, eu, q, tab);
        o = tm.or_put(o, s & 1);
        tm.sync();
        mb = fx_top_bits(tm.or_get(o, s & 1));
        f -= q;
    }
    return d2 == 0 || mb - f <= bound;
}

// Pfaffians of nb node matrices S + wnode[v] D (S packed, m x m, empty modes first, worth
// X 2^-fS, its largest entry of at most mbS bits; D pairs the d leading index pairs), each
// times its node weight and the npo records pvo (the signed pivots of a shared occupied
// elimination, or none); pf[v] of lane seg v is returned on the first lane of the node's
// segment.  Each warp of the team is cut into segments of seg lanes, one per node matrix it
// owns (node v belongs to warp v mod the team's warps); a segment finds the pivot of its
// node's last active row (|g_i| <= sqrt 2 then), inverts it on every lane, moves its index
// to the last but one position and forms the Gauss vectors; the rank-2 updates of all
// nodes are spread over the whole team.  The steps run down to four active indices, whose
// Pfaffian closes the product in three terms, a01 a23 - a02 a13 + a03 a12 (two: a01).
// Returns sum_v gamma[v] prod(pvo) pf(S + wnode[v] D) on thread 0 of the team (NW = 1) or on
// the first lane of each warp its own nodes' sum (NW = 2).
template <class Team>
__device__ inline cd fx_node_pfaffians(const Team &tm, int m, int d, const cd *__restrict__ wnode,
                                       const cd *__restrict__ gamma, int nb, const fx2 *__restrict__ Sx, int fS,
                                       int mbS, fx2 *__restrict__ Ns, int4 *__restrict__ Gv, int4 *__restrict__ Vv,
                                       const uint16_t *__restrict__ tab, fx2 *__restrict__ pv, int *__restrict__ pe,
                                       int npo, const fx2 *__restrict__ pvo, const int *__restrict__ peo) {
    const int npw = (nb + Team::kWarps - 1) / Team::kWarps;  // nodes per warp
    const int seg = npw <= 1 ? 32 : npw <= 2 ? 16 : npw <= 4 ? 8 : 4;
    const int slot = tm.lane / seg, sl = tm.lane - slot * seg;
    const int v = slot * Team::kWarps + tm.wid;
    const bool live = slot < npw && v < nb;
    const int vr = live ? v : 0;  // lanes past the last node read node 0 and write nothing
    const int S0 = m == 0 ? 0 : (m >= 4 ? m / 2 - 1 : 1);  // pivots and the closing Pfaffian
    if (m > 0) {
        const int T = tri_count(m);
        // scale: room for S and for wnode (of modulus one)
        int f = fS;
        if (f > kFxTop || mbS > kFxTop + 1 || mbS < kFxLow) {
            f = fS + kFxTop - mbS;
            f = f < kFxTop ? f : kFxTop;
        }
        if (f == fS) {
            for (int u = tm.t; u < T; u += Team::NT) {
                const fx2 x = Sx[u];
                for (int w = 0; w < nb; ++w) Ns[w * T + u] = x;
            }
        } else {
            for (int u = tm.t; u < T; u += Team::NT) {
                const fx2 x = fx_shift(Sx[u], f - fS);
                for (int w = 0; w < nb; ++w) Ns[w * T + u] = x;
            }
        }
        tm.sync();
        for (int e = tm.t; e < nb * d; e += Team::NT) {
            const int w = e / d, i = e - w * d;
            fx2 *x = Ns + w * T + tri_index(2 * i, 2 * i + 1);
            const fx2 z = fx_of(wnode[w], f);
            *x = make_longlong2(x->x + z.x, x->y + z.y);
        }
        tm.sync();
        fx2 *__restrict__ Nv = Ns + vr * T;
        int mb = kFxTop + 2;
        int s = 0;
        for (int r = m; r > 4; r -= 2, ++s) {
            if (mb > kFxMax || mb < kFxLow) {
                fx_renorm(tm, nb, T, r, Ns, kFxTop - mb);
                f += kFxTop - mb;
                mb = kFxTop;
            }
            // pivot: largest |A_{a,r-1}| of the last row (contiguous entries), each lane
            // scanning every seg-th candidate, then a shuffle reduction in the segment; the
            // key's low bits prefer the first candidate among equal magnitudes
            const fx2 *row = Nv + tri_count(r - 1);
            unsigned bk = 0u;
            for (int a = sl; a < r - 1; a += seg) {
                const unsigned c = ((fx_mag32(row[a]) >> 3) << 6) | (unsigned)(63 - a);
                bk = c > bk ? c : bk;
            }
            for (int o = seg >> 1; o > 0; o >>= 1) {
                const unsigned ob = __shfl_xor_sync(QCS_FULL, bk, o);
                bk = ob > bk ? ob : bk;
            }
            bool zero = false;
            if (__any_sync(QCS_FULL, (bk >> 6) < 64u)) {  // small against the matrix: by the whole words
                bk = 0u;
                for (int a = sl; a < r - 1; a += seg) {
                    const unsigned c = (fx_key(row[a]) << 6) | (unsigned)(63 - a);
                    bk = c > bk ? c : bk;
                }
                for (int o = seg >> 1; o > 0; o >>= 1) {
                    const unsigned ob = __shfl_xor_sync(QCS_FULL, bk, o);
                    bk = ob > bk ? ob : bk;
                }
                zero = (bk >> 6) == 0u;
            }
            const int P = 63 - (int)(bk & 63u);  // 0 .. r - 2
            const fx2 piv = row[P];
            const int rv = r - 2;
            if (live && sl == 0) {
                pv[v * S0 + s] = P != rv ? make_longlong2(-piv.x, -piv.y) : piv;
                pe[v * S0 + s] = f;
            }
            const int sn = zero ? 0 : 61 - fx_bits(piv);
            fxl ir, ii;
            fx_inverse(zero ? make_longlong2(1ll << 60, 0ll) : make_longlong2(piv.x << sn, piv.y << sn), ir, ii);
            if (live) {
                for (int i = sl; i < rv; i += seg) {
                    const bool isP = i == P;
                    const fx2 z = row[isP ? rv : i];
                    // g = A_{i,k} / A_{p,k}, v = A_{i,p}
                    Gv[v * m + i] = zero ? make_int4(0, 0, 0, 0)
                                         : fx_times_inverse(make_longlong2(z.x << sn, z.y << sn), ir, ii);
                    const int o = isP ? rv : i;
                    const fx2 c = P == rv ? Nv[tri_index(i, rv)] : fx_skew(Nv, o, P);
                    Vv[v * m + i] = fx_pack(fx_split(c.x), fx_split(c.y));
                    if (P != rv && !isP) fx_put(Nv, i, P, Nv[tri_index(i, rv)]);
                }
            }
            tm.sync();
            const int q = mb > kFxRoom ? mb - kFxRoom : 0;
            unsigned o = fx_rank2(tm, nb, T, rv, Ns, Gv, Vv, m, 0, q, tab);
            o = tm.or_put(o, s & 1);
            tm.sync();
            mb = fx_top_bits(tm.or_get(o, s & 1));
            f -= q;
        }
        // the closing Pfaffian of the last four (or two) active indices: packed entries
        // 01, 02, 12, 03, 13, 23
        if (live && sl == 0) {
            if (m >= 4) {
                const int sh = kFxTop - mb;
                fxacc re = {0, 0}, im = {0, 0};
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    const fx2 x = fx_shift(Nv[t == 0 ? 0 : t == 1 ? 1 : 3], sh),
                              y = fx_shift(Nv[t == 0 ? 5 : t == 1 ? 4 : 2], sh);
                    fxl xr = fx_split(x.x), xi = fx_split(x.y);
                    const fxl yr = fx_split(y.x), yi = fx_split(y.y);
                    if (t == 1) {
                        xr = fx_neg(xr);
                        xi = fx_neg(xi);
                    }
                    fx_mac(re, xr, yr);
                    fx_mac(re, fx_neg(xi), yi);
                    fx_mac(im, xr, yi);
                    fx_mac(im, xi, yr);
                }
                // |re|, |im| <= 6 2^{116}: kept to 2^{-58} of that
                pv[v * S0 + s] = make_longlong2(fx_value(re, 5), fx_value(im, 5));
                pe[v * S0 + s] = 2 * (f + sh) - 57;
            } else {
                pv[v * S0 + s] = Nv[0];
                pe[v * S0 + s] = f;
            }
        }
    }
    tm.sync();
    // gamma[v] times the records of node v and the npo common ones: each lane of the segment
    // multiplies every seg-th of them, then a shuffle tree over the segment
    fxp z = {1ll << 59, 0, -59};
    bool any = false;
    for (int i = sl; i < S0 + npo + 1; i += seg) {
        fxp y;
        if (i < S0) y = fx_norm(pv[vr * S0 + i], -pe[vr * S0 + i]);
        else if (i < S0 + npo) y = fx_norm(pvo[i - S0], -peo[i - S0]);
        else {
            const cd g = gamma[vr];
            const int E = 1022 - (int)(pivot_key(g) >> 20);
            y = fx_norm(fx_of(g, 58 + E), -(58 + E));
        }
        z = any ? fx_prod(z, y) : y;
        any = true;
    }
    const int w = S0 + npo + 1 < seg ? S0 + npo + 1 : seg;  // lanes that hold a factor
    for (int o = seg >> 1; o > 0; o >>= 1) {
        const fxp y = fx_shfl_xor(z, o);
        if (w > o) z = fx_prod(z, y);  // lanes without a factor hold one
    }
    // sum over the warp's nodes on the segments' first lanes
    cd S = cmk(0.0, 0.0);
    if (live && sl == 0) S = cmk(fx_f64(z.x, z.e), fx_f64(z.y, z.e));
    for (int o = seg; o < 32; o <<= 1) {
        const double sx = __shfl_xor_sync(QCS_FULL, S.x, o), sy = __shfl_xor_sync(QCS_FULL, S.y, o);
        if (o < seg * npw) S = cadd(S, cmk(sx, sy));
    }
    tm.sync();
    return S;
}

// sum_k gamma_k pf(S + wnode_k D) prod(pvo) over nev nodes in rounds of at most NB, on the
// first lane of the team's warps (each its own nodes' part): after a shared elimination
// (shared) of the 2d x 2d complement S, otherwise of the full m x m matrix, one node per
// round.  Ns: NB tri(2d) or tri(m) entries.
template <class Team>
__device__ inline cd fx_node_sum(const Team &tm, int m, int ne, bool shared, int nev, int NB,
                                 const cd *__restrict__ wnode, const cd *__restrict__ gamma, const FxWork &wk,
                                 const fx2 *__restrict__ Sx, int f, int mb, fx2 *__restrict__ Ns,
                                 const uint16_t *__restrict__ tab) {
    cd S = cmk(0.0, 0.0);
    const int mm = shared ? m - ne : m, npo = shared ? ne / 2 : 0, NBr = shared ? NB : 1;
    for (int k0 = 0; k0 < nev; k0 += NBr) {
        const int nb = nev - k0 < NBr ? nev - k0 : NBr;
        const cd s = fx_node_pfaffians(tm, mm, (m - ne) / 2, wnode + k0, gamma + k0, nb, Sx, f, mb, Ns, wk.Gv, wk.Vv,
                                       tab, wk.pv, wk.pe, npo, wk.pv + wk.npv, wk.pe + wk.npv);
        if (tm.lane == 0) S = cadd(S, s);
    }
    return S;
}

// The same from B^(s) in FP64 (packed, in the order of the selection, overwritten): the
// occupied block is eliminated in Ns and S replaces B; a pair for which that is not stable
// takes the full elimination of every node matrix.
template <class Team>
__device__ inline cd fx_pair_sum(const Team &tm, int m, int ne, int nev, int NB, const cd *__restrict__ wnode,
                                 const cd *__restrict__ gamma, const FxWork &wk, cd *Bs, fx2 *Ns,
                                 const uint16_t *__restrict__ tab) {
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    fx2 *Bx = reinterpret_cast<fx2 *>(Bs);
    int f, mb = kFxTop;
    if (!fx_load(tm, m, ne, Bs, Ns, f, tab)) return cmk(nan, nan);
    if (fx_schur_occupied(tm, m, ne, Ns, wk.Gv, wk.Vv, tab, wk.pv + wk.npv, wk.pe + wk.npv, f, mb)) {
        for (int t = tm.t; t < tri_count(m - ne); t += Team::NT) Bx[t] = Ns[t];
        tm.sync();
        return fx_node_sum(tm, m, ne, true, nev, NB, wnode, gamma, wk, Bx, f, mb, Ns, tab);
    }
    tm.sync();
    mb = kFxTop;
    fx_load(tm, m, ne, Bs, Ns, f, tab);
    return fx_node_sum(tm, m, ne, false, nev, 1, wnode, gamma, wk, Ns, f, mb, Bx, tab);
}
