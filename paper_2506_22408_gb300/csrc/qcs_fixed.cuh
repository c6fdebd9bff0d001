// qcs_fixed.cuh -- the Pfaffian eliminations in 64-bit fixed point on the integer pipe.
//
// GB300 issues one 32-lane FP64 FMA per 76 clocks and SM sub-partition, but one 32 x 32 ->
// 64-bit integer multiply-add (IMAD.WIDE) per 4.1 (register-only probes).  A matrix whose
// entries share one power-of-two scale needs no exponent per entry, so the eliminations
// hold every entry as a 64-bit integer X worth X 2^-f, f common to the matrix.  A product
// of two of them takes three IMAD.WIDE on two limbs,
//     X = h 2^S + l,  |l| <= 2^{S-1}:   X Y = hh 2^2S + (h l' + l h') 2^S + l l',
// the last term dropped: 12 to 13 clocks against 76.  With S = 30 and entries of 58 to 60
// bits it is below 2^-58 of the factors' scale, of either sign; longer sums of entries of 57
// bits take S = 29 (2^-60), as S = 31 lost three bits of the congruence against FP64, and of 56
// bits S = 28.  The largest entry of a matrix is kept at 54 to 60 bits, so an update rounds at
// 2^-54 to 2^-60 of it, where FP64 rounds at 2^-53 of each operand: no worse for matrices whose
// entries are of similar size (errors per pair against the oracle, n = 6 to 24, Haar and signed
// permutations, random and near-diagonal walkers: 1.1 to 3.5 10^-15 of the pair scale rms,
// 1.1 to 8.4 10^-15 in FP64, but for n = 8, ne = 4 near-diagonal, 6 10^-15 against 5 10^-14).  An
// entry 2^-k below the largest keeps k bits fewer; where pairs are made of such entries the
// callers leave fixed point (qcs_pairfp64.cuh).
//
// One rank-2 entry update (two complex products) is 24 IMAD.WIDE and about 35 one-clock
// instructions, near 140 clocks per 32 entries, against 8 DFMA = 611 clocks.  With the
// products that cheap, everything around them counts: matrices are ordered with the empty
// modes first and eliminated from the last index up, so that the remaining matrix is a
// prefix of the packed triangle, updated in place without index lists; pivots are compared
// on upper words; products of pivots are taken in normalised fixed point as well.
#pragma once
#include <cmath>

#include "qcs_internal.h"
#include "qcs_ozaki.cuh"
#include "qcs_pair.cuh"

typedef longlong2 fx2;  // complex fixed point, worth (x + i y) 2^-f

// Bits of the largest entry: after a (re)normalisation; before an update at most (limbs of
// 32 bits) and at least.  |g| <= sqrt 2 2^eu and |v| <= sqrt 2 2^mb bound an update by
// 4 2^{mb+eu}: its result is scaled down by q bits when mb + eu exceeds kFxRoom, so that
// it stays below 2^62.4; the scale of the factors themselves is kept, which matters when
// a pivot is small (scaling the matrix down before the update would cost eu bits of g v).
constexpr int kFxTop = 58;
constexpr int kFxMax = 60;
constexpr int kFxLow = 54;
constexpr int kFxRoom = 60;
// Bits by which a multiplier of the occupied elimination may exceed one; pairs beyond take the
// full elimination of every node.  With 20 near-diagonal walkers against signed permutations
// had errors of 7.9 10^-15 rms (n = 12, ne = 6; FP64 2.6 10^-15), with 8 2.1 10^-15.
constexpr int kFxMaxOcc = 8;

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

// A node plan in fixed point: w_k (modulus one) worth X 2^-58, gamma_k worth X 2^ge.
struct FxPlan {
    int nev;
    fx2 w[QCS_MAX_NODES];
    fx2 g[QCS_MAX_NODES];
    int ge[QCS_MAX_NODES];
};

inline void fx_make_plan(const qcs_node_plan &p, FxPlan &q) {
    q.nev = p.nev;
    for (int k = 0; k < p.nev; ++k) {
        q.w[k] = make_longlong2(std::llround(std::ldexp(p.wnode[k].x, 58)), std::llround(std::ldexp(p.wnode[k].y, 58)));
        int e = 0;
        std::frexp(std::fmax(std::fabs(p.gamma[k].x), std::fabs(p.gamma[k].y)), &e);
        q.g[k] = make_longlong2(std::llround(std::ldexp(p.gamma[k].x, 60 - e)),
                                std::llround(std::ldexp(p.gamma[k].y, 60 - e)));
        q.ge[k] = e - 60;
    }
}

struct fxl {  // a fixed-point number as limbs h 2^S + l
    int h, l;
};
template <int S = 30>
__device__ __forceinline__ fxl fx_split(long long X) {
    const unsigned long long y = (unsigned long long)X + (1ull << (S - 1));
    return fxl{(int)__funnelshift_l((unsigned)y, (unsigned)(y >> 32), 32 - S), (int)((unsigned)X << (32 - S)) >> (32 - S)};
}
__device__ __forceinline__ fxl fx_neg(fxl a) { return fxl{-a.h, -a.l}; }

// a b and s + a b in 64 bits, one instruction each: written out because the compiler, when
// it sees a limb's sign extension, multiplies 64-bit numbers with three.
__device__ __forceinline__ long long mul_wide(int a, int b) {
    long long r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ long long mad_wide(int a, int b, long long s) {
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(s));
    return r;
}

struct fxacc {  // hh 2^2S + cr 2^S
    long long hh, cr;
};
// The sum starts at half a unit of its fx_value: a mean over many pairs must not collect the
// half unit that a plain shift loses each time.
__device__ __forceinline__ fxacc fx_mul(fxl a, fxl b, long long half) {
    return fxacc{mul_wide(a.h, b.h), mad_wide(a.l, b.h, mad_wide(a.h, b.l, half))};
}
template <int S = 30>
__device__ __forceinline__ long long fx_half(int dn) {
    return 1ll << (dn - S - 1);
}
__device__ __forceinline__ void fx_mac(fxacc &s, fxl a, fxl b) {
    s.hh = mad_wide(a.h, b.h, s.hh);
    s.cr = mad_wide(a.h, b.l, s.cr);
    s.cr = mad_wide(a.l, b.h, s.cr);
}
// (hh 2^2S + cr 2^S) 2^-dn, S < dn <= 2S
template <int S = 30>
__device__ __forceinline__ long long fx_value(const fxacc &s, int dn) {
    return (s.hh << (2 * S - dn)) + (s.cr >> (dn - S));
}

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

// The same without a branch, |X| < 2^62.
__device__ __forceinline__ long long fx_shift_any(long long X, int s) {
    const int r = s < 0 ? (s > -62 ? -s : 62) : 0;
    const long long y = X << (s > 0 ? s : 0);
    const long long v = (y + ((1ll << r) >> 1)) >> r;
    return s < -62 ? 0ll : v;
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
static __device__ __noinline__ double fx_f64(long long X, int E) {
    bool ok = true;
    const double v = qcs_oz::fixed_to_f64(X, E, ok);
    return ok ? v : qcs_oz::fixed_to_f64_exact(X, E);
}

// 2^118 / (q.x + i q.y) as packed limbs, for max(|q.x|, |q.y|) in [2^59, 2^60): conj(q) / |q|^2,
// the reciprocal R = 2^118 / (|q|^2 2^-60) by one third-order step from the FP32 seed R0
// (relative error e < 2^-22: R = R0 (1 + e + e^2), e^3 < 2^-66) in integers.
__device__ __forceinline__ int4 fx_inverse(fx2 q) {
    const fxl a = fx_split(q.x), b = fx_split(q.y);
    fxacc s = fx_mul(a, a, 0);
    fx_mac(s, b, b);
    const long long D = s.hh + (s.cr >> 30);  // |q|^2 2^-60 in [2^58, 2^61)
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"((float)(int)(D >> 31)));
    const int R0 = (int)(y * 18014398509481984.0f);  // 2^54 y in [2^24, 2^27]
    const long long e = -(long long)((unsigned long long)(unsigned)D * (unsigned)R0 +
                                    ((unsigned long long)((unsigned)(D >> 32) * (unsigned)R0) << 32));  // 2^85 (1 - D R0 2^-85)
    const int eh = (int)(e >> 32);
    const int e2 = __mulhi(eh, eh);
    const long long R = ((long long)R0 << 33) + (mul_wide(R0, eh) >> 20) +
                        (long long)(__umulhi((unsigned)R0, (unsigned)e) >> 20) + (mul_wide(R0, e2) >> 41);
    const fxl r = fx_split(R);
    const fxacc u = fx_mul(a, r, fx_half(60)), v = fx_mul(b, r, fx_half(60));
    return fx_pack(fx_split(fx_value(u, 60)), fx_neg(fx_split(fx_value(v, 60))));
}

// z I 2^-59 for I = 2^118 / q as limbs: 2^59 z / q, as packed limbs.
__device__ __forceinline__ int4 fx_times_inverse(fx2 z, fxl ir, fxl ii) {
    const fxl a = fx_split(z.x), b = fx_split(z.y);
    fxacc re = fx_mul(a, ir, fx_half(59)), im = fx_mul(a, ii, fx_half(59));
    fx_mac(re, fx_neg(b), ii);
    fx_mac(im, b, ir);
    return fx_pack(fx_split(fx_value(re, 59)), fx_split(fx_value(im, 59)));
}

// A complex number (x + i y) 2^e, the larger part of 60 bits (61 at most) unless it is zero.
struct fxp {
    long long x, y;
    int e;
};
__device__ __forceinline__ fxp fx_norm(fx2 a, int e) {
    const unsigned t = fx_mag32(a);
    const int sh = (t ? __clz((int)t) : 64 - fx_bits(a) > 63 ? 4 : 64 - fx_bits(a)) - 4;
    return sh >= 0 ? fxp{a.x << sh, a.y << sh, e - sh} : fxp{a.x >> -sh, a.y >> -sh, e - sh};
}
__device__ __forceinline__ fxp fx_prod(fxp a, fxp b) {
    const fxl ar = fx_split(a.x), ai = fx_split(a.y), br = fx_split(b.x), bi = fx_split(b.y);
    fxacc re = fx_mul(ar, br, fx_half(60)), im = fx_mul(ar, bi, fx_half(60));
    fx_mac(re, fx_neg(ai), bi);
    fx_mac(im, ai, br);
    return fx_norm(make_longlong2(fx_value(re, 60), fx_value(im, 60)), a.e + b.e + 60);
}
__device__ __forceinline__ fxp fx_shfl_xor(const fxp &a, int o) {
    return fxp{__shfl_xor_sync(QCS_FULL, a.x, o), __shfl_xor_sync(QCS_FULL, a.y, o), __shfl_xor_sync(QCS_FULL, a.e, o)};
}

// The Gauss vectors' entries of one index as limbs, g before v.
struct FxGauss {
    int4 g, v;
};

// Rank-2 update, in place, of the leading rv x rv blocks of nb packed matrices (stride T):
//     A_ij = (A_ij + g_i v_j - v_i g_j) 2^-q,   g scaled by 2^{59-eu}.
// Entry t of the packed triangle is read and written by one thread; (i, j) comes from the
// pair table.  Returns this thread's OR of the new entries' upper words.
template <int NT>
__device__ __forceinline__ unsigned fx_rank2(int t0, int nb, int T, int rv, fx2 *__restrict__ Ns,
                                             const FxGauss *__restrict__ GV, int ldv, int eu, int q,
                                             const uint16_t *__restrict__ tab) {
    const int Tr = tri_count(rv), total = nb * Tr;
    const int dn = 59 - eu + q;
    const long long half = fx_half(dn), qhalf = (1ll << q) >> 1;
    unsigned top = 0u;
    int u = t0;
#pragma unroll 1
    for (int e = t0; e < total; e += NT) {
        if (u >= Tr) {  // the next matrix; several for the smallest blocks
            u -= Tr;
            Ns += T;
            GV += ldv;
            if (Tr < NT)
                while (u >= Tr) {
                    u -= Tr;
                    Ns += T;
                    GV += ldv;
                }
        }
        int ia, ib;
        pair_of(tab, u, ia, ib);
        fx2 x = Ns[u];
        const int4 gi = GV[ia].g, vi = GV[ia].v, gj = GV[ib].g, vj = GV[ib].v;
        const fxl gir = {gi.x, gi.y}, gii = {gi.z, gi.w}, gjr = {gj.x, gj.y}, gji = {gj.z, gj.w};
        const fxl vir = {vi.x, vi.y}, vii = {vi.z, vi.w}, vjr = {vj.x, vj.y}, vji = {vj.z, vj.w};
        const fxl mgii = fx_neg(gii), mvir = fx_neg(vir), mvii = fx_neg(vii);
        fxacc re = fx_mul(gir, vjr, half), im = fx_mul(gir, vji, half);
        fx_mac(re, mgii, vji);
        fx_mac(im, gii, vjr);
        fx_mac(re, mvir, gjr);
        fx_mac(im, mvir, gji);
        fx_mac(re, vii, gji);
        fx_mac(im, mvii, gjr);
        if (q > 0) {
            x.x = (x.x + qhalf) >> q;
            x.y = (x.y + qhalf) >> q;
        }
        x.x += fx_value(re, dn);
        x.y += fx_value(im, dn);
        top |= fx_top(x);
        Ns[u] = x;
        u += NT;
    }
    return top;
}

// Multiply the entries of nb packed matrices (tri(r) entries each, stride T) by 2^sh.
template <class Team>
static __device__ __noinline__ void fx_renorm(const Team &tm, int nb, int T, int r, fx2 *Ns, int sh) {
    const int Tr = tri_count(r);
    tm.sync();
    for (int w = 0; w < nb; ++w)
        for (int u = tm.t; u < Tr; u += Team::NT) Ns[w * T + u] = fx_shift(Ns[w * T + u], sh);
    tm.sync();
}

// Records of fx_pair_eliminate's products per warp for NB node matrices per round (vm: the
// entries of the kernel's Gauss-vector buffers, the full matrix or NB complements); the
// ne/2 signed pivots of the shared occupied elimination follow them.  A record is an entry
// worth X 2^-f with its f: 16 + 4 bytes, the f after all the entries.
__host__ __device__ inline int pv_records(int vm, int NB) { return vm / 2 + NB; }
__host__ __device__ inline size_t pv_bytes(int vm, int NB, int ne) {
    return (size_t)(pv_records(vm, NB) + ne / 2) * (sizeof(fx2) + sizeof(int));
}

// Workspace of one pair in the team's shared memory, besides its matrices.
struct FxWork {
    FxGauss *GV;  // Gauss vectors: max(m, NB 2d) entries
    fx2 *pv;      // records
    int *pe;      // ... and their fraction bits
    int npv;      // index of the first occupied pivot's record
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
#pragma unroll 2
    for (int e = tm.lane; e < T; e += 32) {  // every warp of the team takes the maximum itself
        const unsigned k = pivot_key(Bs[e]);
        kb = k > kb ? k : kb;
    }
    kb = __reduce_max_sync(QCS_FULL, kb);
    const int hx = (int)(kb >> 20);  // |x| < 2^{hx - 1022}
    f = kFxTop + 1022 - hx;
    if (hx == 0x7ff) return false;
#pragma unroll 1
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

// x or -x.
__device__ __forceinline__ fx2 fx_neg_if(fx2 x, bool neg) {
    const long long m = neg ? -1ll : 0ll;
    return make_longlong2((x.x ^ m) - m, (x.y ^ m) - m);
}

// Swap of index K with the last of r active ones (K < r - 1) in a packed skew-symmetric
// matrix: the rows' entries change places (each pair by one thread), and the entry between
// the two changes its sign.
template <class Team>
__device__ __forceinline__ void fx_swap_last(const Team &tm, fx2 *__restrict__ N, int r, int K) {
    const int last = tri_count(r - 1), tk = tri_count(K);
#pragma unroll 1
    for (int i = tm.t; i < r - 1; i += Team::NT) {
        const bool lo = i > K;
        fx2 *a = N + (lo ? tri_count(i) + K : tk + i), *b = N + last + i;
        if (i != K) {
            const fx2 x = *a, y = *b;
            *a = fx_neg_if(y, lo);
            *b = fx_neg_if(x, lo);
        } else {
            *b = fx_neg_if(*b, true);
        }
    }
}

// sum_k gamma_k pf(B + w_k D) of one pair, k over the plan's nodes; the sum's parts are on
// the first lanes of the team's warps (each its own nodes).
//
// The node matrices B + w D differ only in their empty x empty block (D pairs the empty
// modes), so eliminating the ne occupied indices first is the same for all of them:
// pf(B + w D) = pf0 pf(S + w D_ee), S the Schur complement of the occupied block.  With
// shared set, job -1 eliminates it in place on X (tri(m) entries worth X 2^-f, the largest of
// at most mb bits, the empty modes first): each step takes the largest entry of the active
// occupied block as pivot (p, k), moves k to the last and p to the last but one position (a
// swap flips the sign) and updates the leading block; S ends as the leading tri(2d)
// entries.  The job fails (ok = false, X overwritten; the caller repeats with a fresh X and
// shared = false) when a pivot is zero, an element of a Gauss vector exceeds 2^kFxMaxOcc or
// the largest entry of S exceeds 2^8 times that of B.
//
// The other jobs are rounds of up to NB node matrices S + w D (one full matrix B + w D per
// round without shared) in Ns.  Each warp of the team is cut into segments of seg lanes,
// one per node matrix it owns (node v belongs to warp v mod the team's warps); a segment
// finds the pivot of its node's last active row (so |g_i| <= sqrt 2), inverts it on every
// lane, moves its index to the last but one position and forms the Gauss vectors; the
// rank-2 updates of all nodes are spread over the whole team.  The steps run down to four
// active indices, whose Pfaffian closes the product in three terms,
// a01 a23 - a02 a13 + a03 a12 (two indices: a01).  Signed pivots, the closing Pfaffian, the
// occupied pivots and gamma are records multiplied by a shuffle tree over the segment.
//
// Both kinds of job run the same step code: one copy keeps the loop in the instruction
// caches (two inlined copies cost the 20-warp kernel 20 % of its issue slots in
// instruction misses).
//
// With kGuard, *lost is set (and ok cleared) when a node's pivot is below 2^-kFxGuard of its
// matrix, or its closing Pfaffian below 2^-(kFxGuard + 6): B is held to 2^-57 of its largest
// entry, so little would be left of such a pair; an occupied pivot that small sends the pair to the
// full elimination.  The records of the product are looked at, not each step's pivot, which took
// 3 % of the steps' time.  Walkers at 10^-2 to 10^-6 from a basis determinant against signed
// permutations (5 and 6 modes) keep 6 10^-11 of a pair's magnitude at worst, 3 10^-10 with
// kFxGuard = 12; a tenth to a half of their pairs is handed over, none of a random walker's.
constexpr int kFxGuard = 10;
template <bool kGuard = false, class Team>
__device__ inline cd fx_pair_eliminate(const Team &tm, int m, int ne, bool shared, int NB, const FxPlan &plan,
                                       const FxWork &wk, fx2 *X, fx2 *Ns, int f, int mb,
                                       const uint16_t *__restrict__ tab, bool &ok, bool *lost = nullptr) {
    const int d2 = m - ne, nev = plan.nev;
    const int bound = mb - f + 8;
    const int mm = shared ? d2 : m, npo = shared ? ne / 2 : 0, NBr = shared ? NB : 1;
    fx2 *pvo = wk.pv + wk.npv;
    int *peo = wk.pe + wk.npv;
    cd total = cmk(0.0, 0.0);
    ok = true;
#pragma unroll 1
    for (int k0 = shared ? -1 : 0; k0 < nev; k0 = k0 < 0 ? 0 : k0 + NBr) {
        const bool occ = k0 < 0;
        const int nb = occ ? 1 : nev - k0 < NBr ? nev - k0 : NBr;
        const int npw = (nb + Team::kWarps - 1) / Team::kWarps;  // nodes per warp
        const int seg = npw <= 1 ? 32 : npw <= 2 ? 16 : npw <= 4 ? 8 : 4;
        const int slot = tm.lane / seg, sl = tm.lane - slot * seg;
        const int v = occ ? 0 : slot * Team::kWarps + tm.wid;
        const bool live = occ || (slot < npw && v < nb);
        const int vr = live ? v : 0;  // lanes past the last node read node 0 and write nothing
        const int mc = occ ? m : mm, T = occ ? 0 : tri_count(mc), stop = occ ? d2 : 4;
        const int S0 = mm == 0 ? 0 : (mm >= 4 ? mm / 2 - 1 : 1);  // a node's pivots and closing Pfaffian
        fx2 *N0 = occ ? X : Ns;  // the job's matrices, stride T
        int fc = f, mbc = mb;
        // pivots below 2^least are refused (w_k has modulus one)
        const int least = (occ || mb > f ? mb - f : 0) - kFxGuard;
        if (!occ && mm > 0) {
            // scale: room for S and for w_k (of modulus one).  A complement of four has no update
            // whose renormalisation would give entries of few bits their place: always scaled.
            mbc = kFxTop + 2;
            if (f > kFxTop || mb > kFxTop + 1 || mb < kFxLow || mm <= 4) {
                fc = f + kFxTop - mb;
                fc = fc < kFxTop ? fc : kFxTop;
                mbc = kFxTop + 1;
            }
#pragma unroll 2
            for (int u = tm.t; u < T; u += Team::NT) {
                fx2 x = X[u];
                if (fc != f) x = fx_shift(x, fc - f);
                for (int w = 0; w < nb; ++w) Ns[w * T + u] = x;
            }
            tm.sync();
            const int d = d2 / 2;
#pragma unroll 1
            for (int e = tm.t; e < nb * d; e += Team::NT) {
                const int w = e / d, i = e - w * d;
                fx2 *x = Ns + w * T + tri_index(2 * i, 2 * i + 1);
                const fx2 z = fx_shift(plan.w[k0 + w], fc - kFxTop);
                *x = make_longlong2(x->x + z.x, x->y + z.y);
            }
            tm.sync();
        }
        fx2 *Nv = N0 + vr * T;
        int s = 0;
#pragma unroll 1
        for (int r = mc; r > stop; r -= 2, ++s) {
            if (mbc > kFxMax || mbc < kFxLow) {
                fx_renorm(tm, nb, T, r, N0, kFxTop - mbc);
                fc += kFxTop - mbc;
                mbc = kFxTop;
            }
            const fx2 *row = Nv + tri_count(r - 1);
            int P, eu = 0;
            bool neg, zero = false;
            if (occ) {
                // the largest entry of the active occupied block (every warp finds it by itself)
                const int ro = r - d2;  // its indices are 2d .. r - 1
                unsigned bk = 0u;
#pragma unroll 1
                for (int t = tm.lane; t < tri_count(ro); t += 32) {
                    int a, b;
                    pair_of(tab, t, a, b);
                    const unsigned c =
                        ((fx_mag32(X[tri_index(d2 + a, d2 + b)]) >> 6) << 9) | (unsigned)(511 - t);
                    bk = c > bk ? c : bk;
                }
                bk = __reduce_max_sync(QCS_FULL, bk);
                int bt = 511 - (int)(bk & 511u);
                if ((bk >> 9) < 64u) {  // small against the matrix: compare by the whole words
                    unsigned kk = 0u, kt = 0u;
#pragma unroll 1
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
                    if (top == 0u) {  // the active occupied block is zero
                        ok = false;
                        return total;
                    }
                    bt = (int)__reduce_min_sync(QCS_FULL, kk == top ? kt : 0xffffffffu);
                }
                int K;
                pair_of(tab, bt, P, K);
                P += d2;
                K += d2;
                neg = false;
                // Every warp has scanned the block before any entry of it is written, here or by
                // the Gauss vectors below: x and -x differ by one in fx_mag32, so a warp that
                // scanned rewritten entries could see another tie and take another pivot.
                tm.sync();
                if (K != r - 1) {
                    fx_swap_last(tm, X, r, K);
                    neg = true;
                    tm.sync();
                }
                // row k can hold larger entries than the pivot among the empty indices
                unsigned rt = 0u;
#pragma unroll 1
                for (int a = tm.lane; a < r - 1; a += 32) rt |= fx_top(row[a]);
                const int rb = fx_top_bits(__reduce_or_sync(QCS_FULL, rt)), pb = fx_bits(row[P]);
                if (rb >= pb) eu = rb - pb + 1;  // |g| 2^-eu < sqrt 2
                if (eu > kFxMaxOcc || (kGuard && pb - fc <= least)) {
                    ok = false;
                    return total;
                }
            } else {
                // the largest of the last row, each lane scanning every seg-th candidate, then a
                // shuffle reduction in the segment; the key's low bits prefer the first
                // candidate among equal magnitudes
                unsigned bk = 0u;
#pragma unroll 1
                for (int a = sl; a < r - 1; a += seg) {
                    const unsigned c = ((fx_mag32(row[a]) >> 3) << 6) | (unsigned)(63 - a);
                    bk = c > bk ? c : bk;
                }
                for (int o = seg >> 1; o > 0; o >>= 1) {
                    const unsigned ob = __shfl_xor_sync(QCS_FULL, bk, o);
                    bk = ob > bk ? ob : bk;
                }
                if (__any_sync(QCS_FULL, (bk >> 6) < 64u)) {  // small against the matrix: by the whole words
                    bk = 0u;
#pragma unroll 1
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
                P = 63 - (int)(bk & 63u);  // 0 .. r - 2
                neg = false;
            }
            const int rv = r - 2;
            const fx2 piv = row[P];
            if (live && (occ ? tm.t : sl) == 0) {
                const int rec = occ ? wk.npv + s : v * S0 + s;
                wk.pv[rec] = fx_neg_if(piv, neg != (P != rv));
                wk.pe[rec] = fc;
            }
            if (r == 2) break;  // no empty modes: the last pivot closes the Pfaffian
            const int sn = zero ? 0 : 60 - fx_bits(piv);
            int4 inv = fx_inverse(zero ? make_longlong2(1ll << 59, 0ll) : make_longlong2(piv.x << sn, piv.y << sn));
            if (zero) inv = make_int4(0, 0, 0, 0);  // a zero row: g = 0, and the product is zero
            if (live) {
                // g_i = A_{i,k} / A_{p,k} scaled by 2^{59-eu}, v_i = A_{i,p}, over the other r - 2
                // positions once what was at the last but one has taken place P: index i reads
                // and writes entries of its own
                const fxl ir = {inv.x, inv.y}, ii = {inv.z, inv.w};
                const int sh = sn - eu, tP = tri_count(P), tL = tri_count(rv);
                const int i0 = occ ? tm.t : sl, step = occ ? Team::NT : seg;
                FxGauss *GV = wk.GV + vr * mc;
#pragma unroll 1
                for (int i = i0; i < rv; i += step) {
                    const int o = i == P ? rv : i;
                    const bool lo = o > P;
                    fx2 *a = Nv + (lo ? tri_count(o) + P : tP + o);
                    fx2 z = row[o];
                    const fx2 y = Nv[tL + i];
                    // P = rv: o = i < P, and y is its own entry (i, P)
                    const fx2 x = fx_neg_if(*a, lo);
                    if (i != P) *a = fx_neg_if(y, lo);
                    if (sh >= 0) {
                        z.x <<= sh;
                        z.y <<= sh;
                    } else {
                        z = fx_shift(z, sh);
                    }
                    GV[i].v = fx_pack(fx_split(x.x), fx_split(x.y));
                    GV[i].g = fx_times_inverse(z, ir, ii);
                }
            }
            tm.sync();
            const int q = mbc + eu > kFxRoom ? mbc + eu - kFxRoom : 0;
            unsigned o = fx_rank2<Team::NT>(tm.t, nb, T, rv, N0, wk.GV, mc, eu, q, tab);
            o = tm.or_put(o, s & 1);
            tm.sync();
            mbc = fx_top_bits(tm.or_get(o, s & 1));
            fc -= q;
        }
        if (occ) {
            if (d2 > 0 && mbc - fc > bound) {
                ok = false;
                return total;
            }
            f = fc;
            mb = mbc;
            tm.sync();
            continue;
        }
        // the closing Pfaffian of the last four (or two) active indices: packed entries
        // 01, 02, 12, 03, 13, 23
        if (mm >= 4) {  // one product on each of the segment's first three lanes
            const int t = sl < 3 ? sl : 0, sh = kFxTop - mbc;
            fx2 x = fx_shift(Nv[t == 2 ? 3 : t], sh);
            const fx2 y = fx_shift(Nv[t == 0 ? 5 : t == 1 ? 4 : 2], sh);
            x = fx_neg_if(x, t == 1);
            const fxl xr = fx_split(x.x), xi = fx_split(x.y), yr = fx_split(y.x), yi = fx_split(y.y);
            fxacc re = fx_mul(xr, yr, fx_half(57)), im = fx_mul(xr, yi, fx_half(57));
            fx_mac(re, fx_neg(xi), yi);
            fx_mac(im, xi, yr);
            // |re|, |im| <= 2 2^{116} each: kept to 2^{-58} of that
            const long long qx = fx_value(re, 57), qy = fx_value(im, 57);
            const long long q1 = __shfl_down_sync(QCS_FULL, qx, 1), q2 = __shfl_down_sync(QCS_FULL, qx, 2);
            const long long p1 = __shfl_down_sync(QCS_FULL, qy, 1), p2 = __shfl_down_sync(QCS_FULL, qy, 2);
            if (live && sl == 0) {
                wk.pv[v * S0 + s] = make_longlong2(qx + q1 + q2, qy + p1 + p2);
                wk.pe[v * S0 + s] = 2 * (fc + sh) - 57;
            }
        } else if (mm > 0 && live && sl == 0) {
            wk.pv[v * S0 + s] = Nv[0];
            wk.pe[v * S0 + s] = fc;
        }
        tm.sync();
        // gamma[v] times the records of node v and the npo common ones: each lane of the segment
        // multiplies every seg-th of them, then a shuffle tree over the segment
        bool tiny = false;
        fxp z = {1ll << 59, 0, -59};
        const int nrec = S0 + npo + 1, w = nrec < seg ? nrec : seg;  // lanes that hold a factor
#pragma unroll 1
        for (int i = sl, o = seg; o > 0;) {
            fxp y;
            bool mul;
            if (i - sl < nrec) {  // uniform over the segment
                mul = i < nrec;
                const bool node = i < S0, po = i < S0 + npo;
                const fx2 *x = !mul || node ? wk.pv + vr * S0 + (mul ? i : 0) : po ? pvo + (i - S0) : plan.g + k0 + vr;
                const int e = !mul ? 0 : node ? -wk.pe[vr * S0 + i] : po ? -peo[i - S0] : plan.ge[k0 + vr];
                if (mul) y = fx_norm(*x, e);
                if (kGuard) tiny |= mul && po && ((y.x | y.y) == 0ll || y.e + 60 <= (i == S0 - 1 ? least - 6 : least));
                i += seg;
            } else {
                o >>= 1;
                if (o == 0) break;
                y = fx_shfl_xor(z, o);
                mul = w > o;  // lanes without a factor hold one
            }
            if (mul) z = fx_prod(z, y);
        }
        if (kGuard) {
            const unsigned t = tm.or_put(tiny, s & 1);
            tm.sync();
            if (tm.or_get(t, s & 1)) {
                ok = false;
                *lost = true;
                return total;
            }
        }
        // sum over the warp's nodes on the segments' first lanes
        cd S = cmk(0.0, 0.0);
        if (live && sl == 0) S = cmk(fx_f64(z.x, z.e), fx_f64(z.y, z.e));
        for (int o = seg; o < 32; o <<= 1) {
            const double sx = __shfl_xor_sync(QCS_FULL, S.x, o), sy = __shfl_xor_sync(QCS_FULL, S.y, o);
            if (o < seg * npw) S = cadd(S, cmk(sx, sy));
        }
        total = cadd(total, S);
        tm.sync();
    }
    return total;
}

// The same from B^(s) in FP64 (packed, in the order of the selection, overwritten by the
// node matrices: max(tri(m), NB tri(2d)) entries); the occupied block is eliminated in X
// (tri(m) entries).  A pair for which that is not stable takes the full elimination of
// every node matrix.
template <class Team>
__device__ inline cd fx_pair_sum(const Team &tm, int m, int ne, int NB, const FxPlan &plan, const FxWork &wk, cd *Bs,
                                 fx2 *X, const uint16_t *__restrict__ tab) {
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    bool shared = true, ok;
    cd S;
#pragma unroll 1
    do {
        int f;
        if (!fx_load(tm, m, ne, Bs, X, f, tab)) return cmk(nan, nan);
        S = fx_pair_eliminate(tm, m, ne, shared, NB, plan, wk, X, reinterpret_cast<fx2 *>(Bs), f, kFxTop, tab, ok);
        shared = false;
        tm.sync();
    } while (!ok);
    return S;
}
