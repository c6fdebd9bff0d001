// qcs_fxsweep.cuh -- inverses of packed skew-symmetric matrices in 64-bit fixed point
// (qcs_fixed.cuh), by sweeps (principal pivot transforms), for the derivatives of Pfaffians.
//
// A sweep on the index pair (p, k) exchanges it between the two sides of y = A x.  With
// a = A_pk, g_i = A_ik / a and v_i = A_ip it keeps A skew-symmetric:
//     A_ij += g_i v_j - v_i g_j,   A_ip = g_i,   A_ik = -v_i / a,   A_pk = -1 / a,
// i and j over every other index, swept or not.  After the sweeps of all pairs A holds its
// inverse; after those of a block P of A = [[C, E], [-E^T, P]] it holds
// [[C + E P^-1 E^T, E P^-1], [.., P^-1]].  One loop of rank-2 updates thus replaces an
// elimination that keeps its factors and the backward recursion over them, at the same
// number of products, and its updates are those of the Pfaffian eliminations.
//
// One common scale would lose the bits of small pivots: swept entries grow like 1/a while
// the others stay.  So each index carries a power of two 2^se, its row and column being
// stored times it (a congruence with a diagonal matrix: every formula above holds for the
// stored entries).  A swept row starts where its entries have 58 bits like the rest of the
// matrix, and any row that exceeds the pivot is shifted down before the update, so that
// |g_i| < 2 sqrt 2: what it loses is small against the update it receives.  Without that
// shift the whole matrix gave up the bits, twice per small pivot, and a mean over 5 10^6
// pairs was 4e-11 off; with it the inverses are 10 to 20 times closer to the exact ones
// than those of an FP64 factorisation.
#pragma once
#include "qcs_fixed.cuh"

struct FxSweepWork {
    FxGauss *GV;       // Gauss vectors: nb mc entries
    fx2 *pv;           // signed pivots: mc/2 of each matrix
    int *pe;           // ... and their fraction bits
    int *bad;          // per matrix: refused
    int *se;           // nb mc: scales of the swept positions
    int8_t *dl;        // nb mc: shifts of one step
    uint8_t *perm;     // nb mc: index that stands at each position
};

constexpr int kFxMaxGrow = 20;  // bits by which a row may exceed the pivot (the callers use FP64 beyond)
constexpr int kFxMaxMult = 3;  // bits of an occupied pivot's multipliers

// Rank-2 update of nb packed matrices of order rest + 2 (stride T), but for the two rows rv and
// rv + 1, g scaled by 2^58:
//     A_ij = A_ij 2^-(dl_i + dl_j) + g_i v_j - v_i g_j.
// Returns this thread's OR of the new entries' upper words.
template <int NT>
__device__ __forceinline__ unsigned fx_sweep_update(int t0, int nb, int T, int rest, int rv, fx2 *__restrict__ Ns,
                                                    const FxGauss *__restrict__ GV, const int8_t *__restrict__ dl,
                                                    const uint16_t *__restrict__ tab) {
    const int Tr = tri_count(rest), total = nb * Tr;
    int u = t0;
    unsigned top = 0u;
#pragma unroll 1
    for (int e = t0; e < total; e += NT) {
        while (u >= Tr) {  // the next matrix
            u -= Tr;
            Ns += T;
            GV += rest + 2;
            dl += rest + 2;
        }
        int ia, ib;
        pair_of(tab, u, ia, ib);
        ia += ia >= rv ? 2 : 0;
        ib += ib >= rv ? 2 : 0;
        fx2 *xp = Ns + tri_count(ib) + ia;
        fx2 x = *xp;
        const int sh = dl[ia] + dl[ib];
        const int4 gi = GV[ia].g, vi = GV[ia].v, gj = GV[ib].g, vj = GV[ib].v;
        const fxl gir = {gi.x, gi.y}, gii = {gi.z, gi.w}, gjr = {gj.x, gj.y}, gji = {gj.z, gj.w};
        const fxl vir = {vi.x, vi.y}, vii = {vi.z, vi.w}, vjr = {vj.x, vj.y}, vji = {vj.z, vj.w};
        const fxl mgii = fx_neg(gii), mvir = fx_neg(vir), mvii = fx_neg(vii);
        fxacc re = fx_mul(gir, vjr, fx_half(58)), im = fx_mul(gir, vji, fx_half(58));
        fx_mac(re, mgii, vji);
        fx_mac(im, gii, vjr);
        fx_mac(re, mvir, gjr);
        fx_mac(im, mvir, gji);
        fx_mac(re, vii, gji);
        fx_mac(im, mvii, gjr);
        if (sh > 0) {
            const long long h = (1ll << sh) >> 1;
            x.x = (x.x + h) >> sh;
            x.y = (x.y + h) >> sh;
        }
        x.x += fx_value(re, 58);
        x.y += fx_value(im, 58);
        top |= fx_top(x);
        *xp = x;
        u += NT;
    }
    return top;
}

struct FxSwept {
    int f, mb, left;  // fraction bits, bits of the largest entry, positions >= stop left unswept
};

// Sweep nb (occ: one) packed matrices of order mc (stride tri(mc), worth X 2^-f, at most mb
// bits) on the positions mc-1 .. stop, two at a time.  occ: the pivot is the largest entry of
// the block of the positions >= stop that are left, its larger index moved to the last one,
// the smaller to the last but one.  Otherwise: the largest entry of the last row, one
// segment of lanes per matrix (matrix v: warp v mod the team's warps).
//
// The occupied sweeps end early, left > 0, when a multiplier of the pivot's column would reach
// 2^kFxMaxMult: an inverse assembled from the blocks loses twice those bits, which a sweep of
// the whole matrix does not.  Limit 3 keeps the gradients' errors below those of the FP64
// code (at 10 to 16 modes one pair in six or seven leaves some indices to the
// nodes); limit 4 was 2 % faster and doubled the largest errors.
//
// mb = -1 when a pivot is below 2^-14 of its matrix or a row exceeds it by more than
// kFxMaxGrow bits (the matrices are overwritten).  Uniform over the team.
template <class Team>
static __device__ __noinline__ FxSwept fx_sweep(Team tm, int mc, int stop, bool occ, int nb, fx2 *N0, int f, int mb,
                                             FxSweepWork wk, const uint16_t *__restrict__ tab) {
    const int T = tri_count(mc), S = (mc - stop) / 2;
    const int npw = (nb + Team::kWarps - 1) / Team::kWarps;
    const int seg = npw <= 1 ? 32 : npw <= 2 ? 16 : npw <= 4 ? 8 : 4;
    const int slot = tm.lane / seg, sl = tm.lane - slot * seg;
    const int v = occ ? 0 : slot * Team::kWarps + tm.wid;
    const bool live = occ || (slot < npw && v < nb);
    const int vr = live ? v : 0;
    const bool lead = live && (occ ? tm.t : sl) == 0;
    fx2 *Nv = N0 + vr * T;
    FxGauss *GV = wk.GV + vr * mc;
    int *se = wk.se + vr * mc;
    int8_t *dl = wk.dl + vr * mc;
    uint8_t *perm = wk.perm + vr * mc;
#pragma unroll 1
    for (int e = tm.t; e < nb * mc; e += Team::NT) {
        const int w = e / mc;
        wk.perm[e] = (uint8_t)(e - w * mc);
        wk.se[e] = 0;
    }
    tm.sync();
    int s = 0;
    unsigned top = 0u;
#pragma unroll 1
    for (int r = mc; r > stop; r -= 2, ++s) {
        if (mb >= kFxMax || mb < kFxTop - 1) {
            fx_renorm(tm, nb, T, mc, N0, kFxTop - mb);
            f += kFxTop - mb;
            mb = kFxTop;
        }
        const int k = r - 1, rv = r - 2;
        fx2 *row = Nv + tri_count(k);
        int P;
        bool neg = false, bad = false;
        if (occ) {
            // the largest entry of the active block (every warp finds it by itself)
            unsigned bk = 0u;
#pragma unroll 1
            for (int t = tm.lane; t < tri_count(r - stop); t += 32) {
                int a, b;
                pair_of(tab, t, a, b);
                const unsigned c = ((fx_mag32(N0[tri_index(stop + a, stop + b)]) >> 6) << 9) | (unsigned)(511 - t);
                bk = c > bk ? c : bk;
            }
            bk = __reduce_max_sync(QCS_FULL, bk);
            int K;
            pair_of(tab, 511 - (int)(bk & 511u), P, K);
            P += stop;
            K += stop;
            const int pb = fx_bits(N0[tri_index(P, K)]);
            unsigned te = 0u;
#pragma unroll 1
            for (int i = tm.lane; i < r; i += 32)
                if (i != P && i != K) te |= fx_top(N0[i < K ? tri_index(i, K) : tri_index(K, i)]);
            // (and a pivot below 2^-10 of the matrix is not told from its neighbours by its key)
            if (fx_top_bits(__reduce_or_sync(QCS_FULL, te)) - pb >= kFxMaxMult || pb < 44) {
                tm.sync();
                return FxSwept{f, mb, r - stop};
            }
            if (K != k) {
                tm.sync();  // every warp has scanned the block
                fx_swap_last(tm, N0, r, K);
#pragma unroll 1
                for (int i = r + tm.t; i < mc; i += Team::NT) {
                    fx2 *x = N0 + tri_count(i);
                    const fx2 y = x[K];
                    x[K] = x[k];
                    x[k] = y;
                }
                if (lead) {
                    const uint8_t u = perm[K];
                    perm[K] = perm[k];
                    perm[k] = u;
                }
                neg = true;
                tm.sync();
            }
        } else {
            // the largest of the last row; the key's low bits prefer the first of equal ones
            unsigned bk = 0u;
#pragma unroll 1
            for (int a = sl; a < k; a += seg) {
                const unsigned c = ((fx_mag32(row[a]) >> 3) << 6) | (unsigned)(63 - a);
                bk = c > bk ? c : bk;
            }
            for (int o = seg >> 1; o > 0; o >>= 1) {
                const unsigned ob = __shfl_xor_sync(QCS_FULL, bk, o);
                bk = ob > bk ? ob : bk;
            }
            P = 63 - (int)(bk & 63u);  // 0 .. r - 2
            bad = (bk >> 6) < 512u;
        }
        const fx2 piv = row[P];
        // bits of column p over every other index
        unsigned tv = 0u;
#pragma unroll 1
        for (int i = occ ? tm.lane : sl; i < mc; i += occ ? 32 : seg)
            if (i != P && i != k) tv |= fx_top(i < P ? Nv[tri_count(P) + i] : Nv[tri_count(i) + P]);
        for (int o = (occ ? 32 : seg) >> 1; o > 0; o >>= 1) tv |= __shfl_xor_sync(QCS_FULL, tv, o);
        const int pb = fx_bits(piv), vb = fx_top_bits(tv);
        if (lead) {
            wk.pv[v * S + s] = fx_neg_if(piv, neg != (P != rv));
            wk.pe[v * S + s] = f;
            wk.bad[v] = bad;
        }
        if (occ) tm.sync();  // both warps have read the columns
        else __syncwarp();
        if (live && !bad) {
            // g scaled by 2^58; stored swept: g 2^57 and (v/a) 2^hk with
            // hk = pb - 1 + min(58 - vb, 1), so that these and (1/a) 2^{57+hk} have at most
            // 59 bits
            const int sn = 60 - pb, lim = vb >= 57 ? 58 - vb : 1;
            const int4 inv = fx_inverse(make_longlong2(piv.x << sn, piv.y << sn));
            const fxl ir = {inv.x, inv.y}, ii = {inv.z, inv.w};
            const int she = sn - 1, shv = 59 - vb, wv = vb - 59 + lim, tP = tri_count(P), tL = tri_count(rv);
            // A_pk = -1/a, by the thread that reads what stood there (or by the leader)
            const fx2 corner =
                fx_shift(make_longlong2(-(((long long)inv.x << 30) + inv.y), -(((long long)inv.z << 30) + inv.w)),
                         lim - 2);
            if (lead) {
                se[rv] = 57 - f;
                se[k] = pb - 1 + lim - f;
                const uint8_t u = perm[P];
                perm[P] = perm[rv];
                perm[rv] = u;
                top |= fx_top(corner);
                if (P == rv) row[rv] = corner;
            }
            // the last but one index takes place P; index i reads and writes entries of its own
#pragma unroll 1
            for (int i = occ ? tm.t : sl; i < mc; i += occ ? Team::NT : seg) {
                if (i == rv || i == k) continue;
                const bool swept = i > k;  // its entries are stored as A_{x,i}
                const int o = i == P ? rv : i, ti = tri_count(i);
                const bool lo = o > P;
                fx2 *a = Nv + (lo ? tri_count(o) + P : tP + o);
                fx2 *zp = swept ? Nv + ti + k : row + o, *yp = swept ? Nv + ti + rv : Nv + tL + i;
                fx2 x = fx_neg_if(*a, lo), z = fx_neg_if(*zp, swept);
                const fx2 y = *yp;
                if (i != P) *a = fx_neg_if(y, lo && !swept);
                else row[rv] = corner;
                // the pivot bounds the other candidates (bits of nearly equal magnitudes can
                // differ): their scales stay, as pivots are recorded without
                int down = swept || i < stop ? fx_bits(z) - pb : 0;
                if (down > 0) {
                    if (down > kFxMaxGrow) wk.bad[v] = 1;
                    x = fx_shift(x, -down);
                    se[i] -= down;
                } else {
                    down = 0;
                }
                dl[i] = (int8_t)down;
                const int4 g = fx_times_inverse(fx_shift(z, she - down), ir, ii);
                const int4 w = fx_times_inverse(fx_shift(x, shv), ir, ii);
                GV[i].g = g;
                GV[i].v = fx_pack(fx_split(x.x), fx_split(x.y));
                const fx2 G = make_longlong2(((((long long)g.x) << 30) + g.y + 1) >> 1,
                                             ((((long long)g.z) << 30) + g.w + 1) >> 1);
                const fx2 W = fx_shift(make_longlong2(((long long)w.x << 30) + w.y, ((long long)w.z << 30) + w.w), wv);
                top |= fx_top(G) | fx_top(W);
                *yp = fx_neg_if(G, swept);
                (swept ? Nv + ti + k : row + i)[0] = fx_neg_if(W, !swept);
            }
        }
        tm.sync();
        for (int w = 0; w < nb; ++w)
            if (wk.bad[w]) return FxSwept{f, -1, 0};
        top |= fx_sweep_update<Team::NT>(tm.t, nb, T, mc - 2, rv, N0, wk.GV, wk.dl, tab);
        top = tm.or_put(top, s & 1);
        tm.sync();
        mb = fx_top_bits(tm.or_get(top, s & 1));
        top = 0u;
    }
    return FxSwept{f, mb, 0};
}

// On the first lane of each matrix's segment (as in fx_sweep): the product of its S pivots,
// npo common records (pvo, peo) and the factor gam[v] 2^ge[v].
template <class Team>
__device__ __forceinline__ cd fx_sweep_product(const Team &tm, int nb, int S, const FxSweepWork &wk, int npo,
                                               const fx2 *pvo, const int *peo, const fx2 *gam, const int *ge, int &v,
                                               bool &lead) {
    const int npw = (nb + Team::kWarps - 1) / Team::kWarps;
    const int seg = npw <= 1 ? 32 : npw <= 2 ? 16 : npw <= 4 ? 8 : 4;
    const int slot = tm.lane / seg, sl = tm.lane - slot * seg;
    v = slot * Team::kWarps + tm.wid;
    const bool live = slot < npw && v < nb;
    const int vr = live ? v : 0;
    lead = live && sl == 0;
    fxp z = {1ll << 59, 0, -59};
    const int nrec = S + npo + 1, w = nrec < seg ? nrec : seg;  // lanes that hold a factor
#pragma unroll 1
    for (int i = sl, o = seg; o > 0;) {
        fxp y;
        bool mul;
        if (i - sl < nrec) {  // uniform over the segment
            mul = i < nrec;
            const bool node = i < S, po = i < S + npo;
            const fx2 *x = !mul || node ? wk.pv + vr * S + (mul ? i : 0) : po ? pvo + (i - S) : gam + vr;
            const int e = !mul ? 0 : node ? -wk.pe[vr * S + i] : po ? -peo[i - S] : ge[vr];
            if (mul) y = fx_norm(*x, e);
            i += seg;
        } else {
            o >>= 1;
            if (o == 0) break;
            y = fx_shfl_xor(z, o);
            mul = w > o;  // lanes without a factor hold one
        }
        if (mul) z = fx_prod(z, y);
    }
    return lead ? cmk(fx_f64(z.x, z.e), fx_f64(z.y, z.e)) : cmk(0.0, 0.0);
}
