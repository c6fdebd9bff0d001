// qcs_grad.cu -- holomorphic walker gradient of the shadow overlap and the force bias.
//
// Per pair the overlap term is pref_w * S_p with S_p = sum_k gamma_k pf(A'_k),
// A'_k = B + conj(z_k) D and B = X J X^T (X = selected rows of the walker-rotated
// snapshot, see qcs_overlap.cu).  Eq. (Pfaffian_der), d pf(A) = pf(A) tr(A^{-1} dA)/2,
// gives dS_p = tr(Y_p dB) with Y_p = (1/2) sum_k gamma_k pf_k A'_k^{-1}, hence
// dS_p = 2 tr(J X^T Y_p dX): the pair's cotangent on X is G_X = 2 Y_p X J.  The
// occupied rows of X are T_j, the empty ones (Re T_j, -Im T_j), T = Ut Qt^T, so
// G_X maps to a holomorphic part on the occupied rows of Ut and an
// antiholomorphic part on its empty rows:
//     Gamma1 += G_X[occ] Qt          (ne x n)
//     Gamma2 += Ht[empty] conj(Qt),  Ht_j = (G_X[2j'] - i G_X[2j'+1]) / 2   (d x n).
// The walker then moves by a unitary rotation of its orbitals (the column
// space part) plus a change of R (the in-span part); with Lambda =
// Gamma1/sqrt2 - U_occ^dagger Gamma2^T U^dagger (the antiholomorphic terms of the
// rotation cancel because the overlap is holomorphic in Phi):
//     g^T = (c0 / P) adj(R) [ S U_occ^dagger + Lambda (I - U_occ U_occ^dagger) ],
//     c0 = 2 i^{ne/2} / 2^{n - ne/2},  S = sum_p S_p,
// with adj(R) = det(R) R^{-1} formed without divisions, so rank-deficient
// walkers need no special case.  The walker rows of Ut are in echelon form
// (qcs_walker.cu): U_occ = U_qr W, and R above is W^H R_qr, so the epilogue
// takes adj(R_qr) det(conj W) W and det(conj W) det(R_qr).
//
// A'_k^{-1} is recomputed per pair and node, never stored in global memory, by sweeps in
// 64-bit fixed point (qcs_fxsweep.cuh): the occupied block, which the node matrices share,
// once per pair; then each node's complement as a whole; then Y_p = sum_k c_k A'_k^{-1} from
// the blocks, which is affine in the complements' inverses (grad_sweeps).  Pairs that the
// sweeps refuse (vanishing pivots, singular node matrices) take an FP64 factorisation and
// backward recursion per node (grad_full_nodes).
#include "qcs_internal.h"
#include "qcs_fxcong.cuh"
#include "qcs_fxsweep.cuh"
#include "qcs_group.cuh"

namespace {

struct GradArgs {
    int n, ne, m, d, nev, NB, nz, nv, all, chunk, nchunks;
    int64_t W, P;
    int group_bytes, tab_bytes;
    int off_Q, off_T, off_NZ, off_g, off_pv, off_pe, off_se, off_perm, off_cf, off_invh, off_hist, off_scr;
    const cd *Ut;
    const cd *Qh;        // per snapshot of the set: the rows [H1^T; G2^T] (2n x n, the layout of Qt)
    const int *idx;
    const int *d_count;
    cd *partial;
    unsigned long long *counter;  // tile counter: groups pull tiles dynamically
    unsigned *status;
    FxPlan plan;
    cd wnode[QCS_MAX_NODES];
    cd gamma[QCS_MAX_NODES];
};

struct GradShared {  // per-group scalars exchanged between the two warps
    unsigned red[4];
    int bad[kMaxNBG], pos;
    long long slot;
    cd pf;
};

// Y = (1/2) sum_k gamma_k pf_k A'_k^{-1} in FP64, every node matrix factored and inverted in
// full, for pairs that the fixed-point sweeps refuse (small pivots, singular matrices).
// Bs: B^(s), the occupied rows first.  Returns S_p on thread 0.
static __device__ __noinline__ cd grad_full_nodes(const GradArgs &A, const cd *Bs, cd *Ys, cd *Ns, unsigned char *wb,
                                                  const uint16_t *tab, int t, int bar) {
    const int m = A.m, T = tri_count(m);
    cd *vec = reinterpret_cast<cd *>(wb + A.off_g), *invh = reinterpret_cast<cd *>(wb + A.off_invh);
    uint8_t *acth = wb + A.off_hist, *kh = acth + (m / 2 + 1) * m, *ph = kh + m / 2;
    GradShared *scr = reinterpret_cast<GradShared *>(wb + A.off_scr);
    cd S = cmk(0.0, 0.0);
    for (int e = t; e < T; e += kGroup) Ys[e] = cmk(0.0, 0.0);
    group_sync(bar);
    for (int k = 0; k < A.nev; ++k) {
        node_factor(m, A.ne, A.wnode + k, 1, Bs, Ns, vec, vec + m, &scr->pf, invh, &scr->pos, acth, kh, ph, tab, t, bar,
                    A.status);
        node_inverse(m, 1, Ns, vec, vec + m, vec + 2 * m, vec + 3 * m, invh, acth, kh, ph, t, bar);
        const cd c = cmul(A.gamma[k], scr->pf), h = cscale(c, 0.5);
        S = cadd(S, c);
        for (int e = t; e < T; e += kGroup) {
            cd y = Ys[e];
            cfma(y, h, Ns[e]);
            Ys[e] = y;
        }
        group_sync(bar);
    }
    return S;
}

// The same by fixed-point sweeps (qcs_fxsweep.cuh), from B^(s) in X (empties first, worth
// X 2^-f, at most mb bits; overwritten).  The node matrices differ only in their empty x
// empty block, so with the occupied block P swept once (all of it but for pairs of small
// pivots, which stay with the empty modes' rows),
//     [[C, E], [-E^T, Pi]],   C the Schur complement, E = B_eo P^-1, Pi = P^-1,
// and Z_k = (C + w_k D)^-1 by one sweep of a whole matrix per node,
//     A'_k^{-1} = [[Z_k, -Z_k E], [-E^T Z_k, Pi + E^T Z_k E]],
// which is affine in Z_k: one assembly from Zc = sum_k c_k Z_k, c_k = gamma_k pf_k / 2.
// Returns false (uniform over the group) when a sweep is refused or C exceeds 2^8 times B;
// S = S_p on every thread.
static __device__ __noinline__ bool grad_sweeps(const GradArgs &A, fx2 *X, cd *Ys, fx2 *Ns, unsigned char *wb, int f,
                                                int mb, cd &S, const uint16_t *tab, int t, int bar) {
    const int m = A.m, ne = A.ne, d2 = m - ne;
    GradShared *scr = reinterpret_cast<GradShared *>(wb + A.off_scr);
    const FxTeam<2> tm = {t, t & 31, t >> 5, bar, scr->red};
    FxGauss *GV = reinterpret_cast<FxGauss *>(wb + A.off_g);
    fx2 *pv = reinterpret_cast<fx2 *>(wb + A.off_pv);
    int *pe = reinterpret_cast<int *>(wb + A.off_pe), *seo = reinterpret_cast<int *>(wb + A.off_se);
    uint8_t *permo = wb + A.off_perm, *at = permo + m + A.nv;  // at: position of each index, per node
    int8_t *dl = reinterpret_cast<int8_t *>(at + A.nv);
    cd *cf = reinterpret_cast<cd *>(wb + A.off_cf);
    const FxSweepWork wo = {GV, pv, pe, scr->bad, seo, dl, permo};
    const FxSweepWork wn = {GV, pv + ne / 2, pe + ne / 2, scr->bad, seo + m, dl, permo + m};
    const int bound = mb - f + 8;
    const FxSwept o = fx_sweep(tm, m, d2, true, 1, X, f, mb, wo, tab);
    if (o.mb < 0) return false;
    f = o.f;
    // rows and columns of C: md positions; of Pi: no
    const int md = d2 + o.left, no = ne - o.left, npo = no / 2, Tn = tri_count(md);
    // selected row at position x
    auto sel = [&](int x) { return x < d2 ? ne + x : permo[x] - d2; };
    auto put = [&](int x, int y, cd v) {  // A^-1 at positions (x, y), to selected rows
        const int a = sel(x), b = sel(y);
        Ys[a < b ? tri_index(a, b) : tri_index(b, a)] = flip_if(v, a > b);
    };
    // scales of C (room for w_k, of modulus one) and E
    int sb = -0x10000, eb = -0x10000;
    for (int e = t; e < Tn; e += kGroup) {
        int a, b;
        pair_of(tab, e, a, b);
        sb = max(sb, fx_bits(X[e]) - seo[a] - seo[b]);
        put(a, b, cmk(0.0, 0.0));
    }
    for (int e = t; e < md * no; e += kGroup) {
        const int c = e / md, i = e - c * md;
        eb = max(eb, fx_bits(X[tri_index(i, md + c)]) - seo[i]);
    }
    sb = __reduce_max_sync(QCS_FULL, sb);
    eb = __reduce_max_sync(QCS_FULL, eb);
    group_sync(bar);
    if (tm.lane == 0) {
        scr->red[tm.wid] = (unsigned)sb;
        scr->red[2 + tm.wid] = (unsigned)eb;
    }
    group_sync(bar);
    sb = max((int)scr->red[0], (int)scr->red[1]);
    eb = max((int)scr->red[2], (int)scr->red[3]);
    if (md > 0 && sb - f > bound) return false;
    int fn = f + kFxTop - sb;
    fn = fn < kFxTop ? fn : kFxTop;
    int NB = A.NB;
    if (md > d2) {
        if (NB * Tn > A.nz) NB = A.nz / Tn;
        if (NB * md > A.nv) NB = A.nv / md;
    }
    cd csum = cmk(0.0, 0.0);
#pragma unroll 1
    for (int k0 = 0; k0 < A.nev; k0 += NB) {
        const int nb = A.nev - k0 < NB ? A.nev - k0 : NB;
        FxSwept z = {0, 0, 0};
        if (md > 0) {
#pragma unroll 1
            for (int e = t; e < Tn; e += kGroup) {
                int a, b;
                pair_of(tab, e, a, b);
                const fx2 x = fx_shift(X[e], fn - f - seo[a] - seo[b]);
                const bool dd = (a & 1) == 0 && b == a + 1 && b < d2;
                for (int w = 0; w < nb; ++w) {
                    fx2 y = x;
                    if (dd) {
                        const fx2 d = fx_shift(A.plan.w[k0 + w], fn - kFxTop);
                        y = make_longlong2(x.x + d.x, x.y + d.y);
                    }
                    Ns[w * Tn + e] = y;
                }
            }
            z = fx_sweep(tm, md, 0, false, nb, Ns, fn, kFxTop + 1, wn, tab);
            if (z.mb < 0) return false;
        }
        int v;
        bool lead;
        const cd c = fx_sweep_product(tm, nb, md / 2, wn, npo, pv, pe, A.plan.g + k0, A.plan.ge + k0, v, lead);
        if (lead) cf[v] = cscale(c, 0.5);
        for (int e = t; e < nb * md; e += kGroup) {
            const int w = e / md;
            at[w * md + wn.perm[e]] = (uint8_t)(e - w * md);
        }
        group_sync(bar);
        for (int w = 0; w < nb; ++w) csum = cadd(csum, cf[w]);
#pragma unroll 1
        for (int e = t; e < Tn; e += kGroup) {
            int a, b;
            pair_of(tab, e, a, b);
            cd y = cmk(0.0, 0.0);
#pragma unroll 1
            for (int w = 0; w < nb; ++w) {
                const int i = at[w * md + a], j = at[w * md + b];
                const fx2 x = fx_neg_if(Ns[w * Tn + (i < j ? tri_index(i, j) : tri_index(j, i))], i > j);
                const int E = -z.f - wn.se[w * md + i] - wn.se[w * md + j];
                cfma(y, cf[w], cmk(fx_f64(x.x, E), fx_f64(x.y, E)));
            }
            put(a, b, k0 == 0 ? y : cadd(y, skew_at(Ys, sel(a), sel(b))));
        }
        group_sync(bar);
    }
    S = cscale(csum, 2.0);
    if (no == 0) return true;
    // F = Zc E (worth F 2^{-fF - se_c} in column c)
    unsigned kz = 0u;
    for (int e = t; e < Tn; e += kGroup) {
        int a, b;
        pair_of(tab, e, a, b);
        kz = max(kz, pivot_key(skew_at(Ys, sel(a), sel(b))));
    }
    kz = __reduce_max_sync(QCS_FULL, kz);
    if (tm.lane == 0) scr->red[tm.wid] = kz;
    group_sync(bar);
    kz = max(scr->red[0], scr->red[1]);
    if (kz >= 0x7ff00000u) return false;
    const int fz = fx_fraction(kz, 56), fE = f + 56 - eb;
    const int dn = 51 + (md > 1 ? 32 - __clz(md - 1) : 0);  // md products of 2^113 stay below 2^63
    int4 *Zl = reinterpret_cast<int4 *>(Ns), *El = Zl + Tn, *Fl = El + md * no;
    for (int e = t; e < Tn; e += kGroup) {
        int a, b;
        pair_of(tab, e, a, b);
        Zl[e] = fx_limbs(skew_at(Ys, sel(a), sel(b)), fz);
    }
    for (int e = t; e < md * no; e += kGroup) {
        const int c = e / md, i = e - c * md;
        const fx2 x = fx_shift(X[tri_index(i, md + c)], 56 - eb - seo[i]);
        El[e] = fx_pack(fx_split<kFxS>(x.x), fx_split<kFxS>(x.y));
    }
    group_sync(bar);
    unsigned top = 0u;
#pragma unroll 1
    for (int e = t; e < md * no; e += kGroup) {
        const int c = e / md, i = e - c * md;
        const int4 *er = El + c * md, *zr = Zl + tri_count(i);
        fxacc p1 = {0, 0}, p2 = {0, 0}, p3 = {0, 0};
#pragma unroll 1
        for (int j = 0; j < md; ++j) {
            if (j == i) {  // below: -Z_ij = Z_ji; from here on Z_ij
                p1 = fx_accsub(fxacc{0, 0}, p1);
                p2 = fx_accsub(fxacc{0, 0}, p2);
                p3 = fx_accsub(fxacc{0, 0}, p3);
                continue;
            }
            const int4 z = j < i ? zr[j] : Zl[tri_count(j) + i], x = er[j];
            fx_mac(p1, fx_re(z), fx_re(x));
            fx_mac(p2, fx_im(z), fx_im(x));
            fx_mac(p3, fx_add(fx_re(z), fx_im(z)), fx_add(fx_re(x), fx_im(x)));
        }
        fxacc re = fx_accsub(p1, p2), im = fx_accsub(fx_accsub(p3, p1), p2);
        re.cr += fx_half<kFxS>(dn);
        im.cr += fx_half<kFxS>(dn);
        const fx2 F = make_longlong2(fx_value<kFxS>(re, dn), fx_value<kFxS>(im, dn));
        top |= fx_top(F);
        X[tri_index(i, md + c)] = F;
    }
    top = tm.or_put(top, 1);
    group_sync(bar);
    const int fb = fx_top_bits(tm.or_get(top, 1)), fF = fz + fE - dn;
#pragma unroll 1
    for (int e = t; e < md * no; e += kGroup) {
        const int c = e / md, i = e - c * md;
        const fx2 F = X[tri_index(i, md + c)], x = fx_shift(F, 56 - fb);
        Fl[e] = fx_pack(fx_split<kFxS>(x.x), fx_split<kFxS>(x.y));
        const int E = -fF - seo[md + c];
        put(i, md + c, cmk(-fx_f64(F.x, E), -fx_f64(F.y, E)));
    }
    group_sync(bar);
    const int fP = fE + fF + 56 - fb - dn;
#pragma unroll 1
    for (int e = t; e < tri_count(no); e += kGroup) {
        int c, c2;
        pair_of(tab, e, c, c2);
        fxacc p1 = {0, 0}, p2 = {0, 0}, p3 = {0, 0};
#pragma unroll 1
        for (int i = 0; i < md; ++i) {
            const int4 z = El[c * md + i], x = Fl[c2 * md + i];
            fx_mac(p1, fx_re(z), fx_re(x));
            fx_mac(p2, fx_im(z), fx_im(x));
            fx_mac(p3, fx_add(fx_re(z), fx_im(z)), fx_add(fx_re(x), fx_im(x)));
        }
        fxacc re = fx_accsub(p1, p2), im = fx_accsub(fx_accsub(p3, p1), p2);
        re.cr += fx_half<kFxS>(dn);
        im.cr += fx_half<kFxS>(dn);
        const int sc = seo[md + c] + seo[md + c2];
        const fx2 pi = X[tri_index(md + c, md + c2)];
        cd y = cmul(csum, cmk(fx_f64(pi.x, -f - sc), fx_f64(pi.y, -f - sc)));
        y.x += fx_f64(fx_value<kFxS>(re, dn), -fP - sc);
        y.y += fx_f64(fx_value<kFxS>(im, dn), -fP - sc);
        put(md + c, md + c2, y);
    }
    group_sync(bar);
    return true;
}

// Two warps (a group of 64 threads) per pair; a block holds blockDim/64 groups,
// each with its own workspace and named barrier.  Groups pull (walker, chunk)
// tiles from a device counter in chunk-major order.
//
// In FP64 a pair at 16 modes and 8 electrons took 190k operations on a pipe that issues 32
// lanes per 76 clocks: 606 ms for 512 walkers against 10,000 snapshots.  K, B^(s) and the
// cotangent products as two-limb integers: 490 ms.  The inverses by fixed-point sweeps:
// 343 ms, now 33k instructions a pair at an issue rate of 45 %, bound by latency (dependent
// multiply-adds, pivot searches and the barriers of each sweep step).  Of that, K and B take
// a seventh, the occupied sweeps a sixth, the nodes a third, the assembly of Y a fifth and
// the cotangents a sixth.  Four blocks of two groups per SM (128 registers, 28 KB a group:
// Y in the walker rows' place, which are staged anew for each pair, and the cotangents
// accumulated in global memory) against three: 1.03x, 1.08x at 10 modes.
__global__ void __launch_bounds__(128, 4) grad_pair_kernel(const __grid_constant__ GradArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gid = threadIdx.x / kGroup;
    const int t = threadIdx.x - gid * kGroup;
    const int bar = 1 + gid;
    const int n = A.n, n2 = 2 * n, ne = A.ne, m = A.m, T = tri_count(m);
    const int lt = ld_t(n);
    // the pair table and the groups' workspaces fit the launch's shared memory
    if (!QCS_IN_BOUNDS(T * (int)sizeof(uint16_t) <= A.tab_bytes &&
                           (size_t)A.tab_bytes + (size_t)(blockDim.x / kGroup) * A.group_bytes <= dyn_smem_bytes(),
                       A.status))
        return;
    uint16_t *tab = reinterpret_cast<uint16_t *>(smem_raw);
    build_pair_table(tab, T);
    __syncthreads();
    unsigned char *wb = smem_raw + A.tab_bytes + (size_t)gid * A.group_bytes;
    int4 *Us = reinterpret_cast<int4 *>(wb);             // walker rows as limbs (qcs_fxcong.cuh)
    int4 *Qs = reinterpret_cast<int4 *>(wb + A.off_Q);   // half of the snapshot's rows as limbs
    fx2 *Xs = reinterpret_cast<fx2 *>(wb + A.off_Q);     // B^(s) in fixed point, once K is formed
    int4 *Ks = reinterpret_cast<int4 *>(wb + A.off_T);   // K as limbs
    cd *Ys = reinterpret_cast<cd *>(wb);  // in the walker rows' place, once B^(s) is formed
    cd *Ns = reinterpret_cast<cd *>(wb + A.off_NZ);  // node matrices, then their inverses, then the coefficients
    GradShared *scr = reinterpret_cast<GradShared *>(wb + A.off_scr);

    const int64_t L = A.all ? A.P : (int64_t)(*A.d_count);
    const int64_t ntiles = A.W * A.nchunks;
    const size_t rec = 1 + (size_t)n * n;
    for (;;) {
        if (t == 0) scr->slot = (long long)atomicAdd(A.counter, 1ull);
        group_sync(bar);
        const int64_t tile = (int64_t)scr->slot;  // rewritten only after the barriers below
        if (tile >= ntiles) break;
        const int ch = (int)(tile / A.W);  // chunk-major: a snapshot chunk is fetched once
        const int64_t w = tile - (int64_t)ch * A.W;
        const int64_t p0 = (int64_t)ch * A.chunk;
        const int64_t p1 = p0 + A.chunk < L ? p0 + A.chunk : L;
        if (!QCS_IN_BOUNDS(ch < A.nchunks && L >= 0 && L <= A.P, A.status)) {  // group-uniform
            group_sync(bar);  // every thread has read the slot before it is rewritten
            continue;
        }
        cd *out = A.partial + (w * A.nchunks + ch) * rec, *Gs = out + 1;  // entry e: thread e mod 64
        cd Ssum = cmk(0.0, 0.0);
        for (int e = t; e < n * n; e += kGroup) Gs[e] = cmk(0.0, 0.0);
        if (p0 < L) {
            const cd *Utw = A.Ut + w * n * n;
            const int fU = fx_fraction(fx_max_key(Utw, n * n, t & 31), 57);
            for (int64_t pq = p0; pq < p1; ++pq) {
                const int64_t q = A.all ? pq : (int64_t)A.idx[pq];
                if (!QCS_IN_BOUNDS(q >= 0 && q < A.P, A.status)) continue;  // group-uniform
                group_sync(bar);
                // K = Ut [H1 | G2] by column halves, then B^(s) from it, in fixed point
                const cd *Qr = A.Qh + q * n2 * n;
                const unsigned key = fx_max_key(Qr, n2 * n, t & 31);
                if (key >= 0x7ff00000u) {  // a non-finite snapshot (every snapshot evaluated): NaN
                    const double nan = __longlong_as_double(0x7ff8000000000000ll);
                    for (int e = t; e < n * n; e += kGroup) Gs[e] = cmk(nan, nan);
                    if (t == 0) {
                        raise_status(A.status, QCS_ERR_NONFINITE);
                        Ssum = cmk(nan, nan);
                    }
                    continue;
                }
                const int fQ = fx_fraction(key, 57);
                const FxTeam<2> tm = {t, t & 31, t >> 5, bar, scr->red};
                unsigned top = 0u;
                fx_stage_rows(n, n * n, Utw, fU, nullptr, Us, t, kGroup);
                for (int h = 0; h < 2; ++h) {
                    fx_stage_rows(n, n * n, Qr + (int64_t)h * n * n, fQ, nullptr, Qs, t, kGroup);
                    group_sync(bar);
                    top |= fx_build_T(n, ne, Us, Qs, reinterpret_cast<fx2 *>(Ks), h * n, t, kGroup);
                    group_sync(bar);
                }
                top = tm.or_put(top, 0);
                group_sync(bar);
                const int kb = fx_top_bits(tm.or_get(top, 0));
                const int fK = fU + fQ - 58 + 56 - kb;
                fx_T_limbs<kFxS>(n, Ks, kb, t, kGroup);
                group_sync(bar);
                top = tm.or_put(fx_build_B_from_K(n, ne, Us, Ks, Xs, tab, t, kGroup), 1);
                group_sync(bar);
                const int fB = fK + fU - 58;
                cd S;
                if (!grad_sweeps(A, Xs, Ys, reinterpret_cast<fx2 *>(Ns), wb, fB, fx_top_bits(tm.or_get(top, 1)), S, tab,
                                 t, bar)) {
                    group_sync(bar);
                    fx_stage_rows(n, n * n, Utw, fU, nullptr, Us, t, kGroup);
                    group_sync(bar);
                    fx2 *Bx = reinterpret_cast<fx2 *>(Ns);
                    cd *Bs = reinterpret_cast<cd *>(Xs);
                    fx_build_B_from_K(n, ne, Us, Ks, Bx, tab, t, kGroup);
                    group_sync(bar);
                    for (int e = t; e < T; e += kGroup) {  // to FP64, the occupied rows first
                        int a, b;
                        pair_of(tab, e, a, b);
                        const int i = a < m - ne ? a + ne : a - (m - ne), j = b < m - ne ? b + ne : b - (m - ne);
                        const cd v = flip_if(cmk(fx_f64(Bx[e].x, -fB), fx_f64(Bx[e].y, -fB)), i > j);
                        Bs[i < j ? tri_index(i, j) : tri_index(j, i)] = v;
                    }
                    group_sync(bar);
                    S = grad_full_nodes(A, Bs, Ys, Ns, wb, tab, t, bar);
                }
                if (t == 0) {
                    if (!cfinite(S)) raise_status(A.status, QCS_ERR_NONFINITE);
                    Ssum = cadd(Ssum, S);
                }
                // Cotangents: Gamma1 (rows < ne) += G_X[occ] Qt and Gamma2 (rows >= ne) += Ht conj(Qt),
                // G_X / 2 = Y (X J) and Ht_i = G[ne+2i] - i G[ne+2i+1] = Yh_i (X J), where
                // Yh_i = Y[ne+2i] - i Y[ne+2i+1] (G_X is linear in Y's rows).  X J Qt and
                // X J conj(Qt) are rows of K = [Ut H1 | Ut G2]: occupied row b gives K1_b and
                // K2_b; the empty rows R_j, I_j give (K1_j + conj K2_j)/2, i (K1_j - conj K2_j)/2
                // and their conjugates.  So with the source row y (Y[r] for r < ne, Yh_{r-ne} else)
                // and c_j = (y[R_j] + i y[I_j])/2, c'_j = (y[R_j] - i y[I_j])/2,
                //     Gamma1[r] += sum_b y[b] K1_b + sum_j (c_j K1_j + c'_j conj K2_j)
                //     Gamma2[r] += sum_b y[b] K2_b + sum_j (c_j K2_j + c'_j conj K1_j)
                // (n x m coefficients Cf in the node region, as limbs once their largest is
                // known, then n x n entries of m terms, three real products each: with the
                // sums of K's parts (differences for the conjugated ones), Re = p1 - p2 and
                // Im = p3 - p1 - p2).
                cd *Cf = Ns;
                unsigned ck = 0u;
                for (int e = t; e < n * m; e += kGroup) {
                    const int r = e / m, b = e - r * m;
                    const bool occ = r < ne;
                    const int r0 = occ ? r : ne + 2 * (r - ne), r1 = occ ? r : r0 + 1;
                    const bool pair = b >= ne;
                    const int b0 = pair ? ne + ((b - ne) & ~1) : b;
                    // y at columns b0 and bi = b0 + 1 (the second only for an empty pair)
                    const int bi = pair ? b0 + 1 : b0;
                    cd y0 = skew_at(Ys, r0, b0), y1 = skew_at(Ys, r1, b0);
                    const cd yb = occ ? y0 : cmk(y0.x + y1.y, y0.y - y1.x);
                    y0 = skew_at(Ys, r0, bi);
                    y1 = skew_at(Ys, r1, bi);
                    const cd yi = occ ? y0 : cmk(y0.x + y1.y, y0.y - y1.x);
                    // c = (yb + i yi) / 2 at even offsets, c' = (yb - i yi) / 2 at odd ones
                    const bool odd = (b - ne) & 1;
                    const cd iy = flip_if(cmk(-yi.y, yi.x), odd);
                    const cd c = pair ? cmk(0.5 * (yb.x + iy.x), 0.5 * (yb.y + iy.y)) : yb;
                    Cf[e] = c;
                    ck = max(ck, pivot_key(c));
                }
                ck = __reduce_max_sync(QCS_FULL, ck);
                if ((t & 31) == 0) scr->red[t >> 5] = ck;
                group_sync(bar);
                ck = max(scr->red[0], scr->red[1]);
                if (ck >= 0x7ff00000u) {  // an overflowed inverse: NaN, as its products would be
                    const double nan = __longlong_as_double(0x7ff8000000000000ll);
                    for (int e = t; e < n * n; e += kGroup) Gs[e] = cmk(nan, nan);
                    continue;
                }
                const int fC = fx_fraction(ck, 56);
                int4 *Cx = reinterpret_cast<int4 *>(Cf);
                for (int e = t; e < n * m; e += kGroup) Cx[e] = fx_limbs(Cf[e], fC);
                group_sync(bar);
#pragma unroll 1
                for (int e = t; e < n * n; e += kGroup) {
                    const int r = e / n, k = e - r * n;
                    const int o1 = r < ne ? 0 : n, o2 = n - o1;
                    const int4 *cf = Cx + r * m, *kr = Ks + k;
                    fxacc p1 = {0, 0}, p2 = {0, 0}, p3 = {0, 0};
#pragma unroll 1
                    for (int b = 0; b < ne; ++b, kr += lt) {
                        const int4 c = cf[b], v = kr[o1];
                        fx_mac(p1, fx_re(c), fx_re(v));
                        fx_mac(p2, fx_im(c), fx_im(v));
                        fx_mac(p3, fx_add(fx_re(c), fx_im(c)), fx_add(fx_re(v), fx_im(v)));
                    }
                    cf += ne;
#pragma unroll 1
                    for (int j = 0; j < A.d; ++j, kr += lt, cf += 2) {
                        const int4 c = cf[0], v = kr[o1], c2 = cf[1], w2 = kr[o2];  // c v + c2 conj(w2)
                        fx_mac(p1, fx_re(c), fx_re(v));
                        fx_mac(p2, fx_im(c), fx_im(v));
                        fx_mac(p3, fx_add(fx_re(c), fx_im(c)), fx_add(fx_re(v), fx_im(v)));
                        fx_mac(p1, fx_re(c2), fx_re(w2));
                        fx_mac(p2, fx_neg(fx_im(c2)), fx_im(w2));
                        fx_mac(p3, fx_add(fx_re(c2), fx_im(c2)), fx_sub(fx_re(w2), fx_im(w2)));
                    }
                    fxacc re = fx_accsub(p1, p2), im = fx_accsub(fx_accsub(p3, p1), p2);
                    re.cr += fx_half<kFxS>(58);
                    im.cr += fx_half<kFxS>(58);
                    const cd acc = Gs[e];
                    Gs[e] = cmk(acc.x + fx_f64(fx_value<kFxS>(re, 58), 58 - fC - fK),
                                acc.y + fx_f64(fx_value<kFxS>(im, 58), 58 - fC - fK));
                }
            }
        }
        group_sync(bar);
        if (t == 0) out[0] = Ssum;
    }
}

// Per walker: sum the tile records in order, then
//   O = c0 det(R) S / P,   g^T = (c0/P) adj(R) [S U_occ^dagger + Lambda (I - U_occ U_occ^dagger)],
//   Lambda = sqrt2 Gacc1 - U_occ^dagger Gacc2^T U^dagger
// where Gacc1 = Gamma1 / 2 and Gacc2 = Gamma2 as accumulated by grad_pair_kernel.
__global__ void grad_epilogue_kernel(int n, int ne, int64_t W, int64_t P, int nchunks, const cd *__restrict__ partial,
                                     const cd *__restrict__ U, const cd *__restrict__ R,
                                     const cd *__restrict__ Wrot, cd *__restrict__ overlap,
                                     cd *__restrict__ grad, unsigned *status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int nn = n * n;
    cd *G = reinterpret_cast<cd *>(smem_raw) + (size_t)warp * (4 * nn + 2 * ne * n + 2 * ne * ne + 2);
    cd *Us = G + nn;           // U (n x n)
    cd *V1 = Us + nn;          // Gamma2^T U^dagger (n x n)
    cd *Lm = V1 + nn;          // Lambda (ne x n)
    cd *Mm = Lm + ne * n;      // S U_occ^dagger + Lambda'  (ne x n)
    cd *Rs = Mm + ne * n;      // R (ne x ne)
    cd *Ad = Rs + ne * ne;     // adj(R)
    cd *Sv = Ad + ne * ne;     // S
    const double sq2 = 1.41421356237309504880;
    const size_t rec = 1 + (size_t)nn;
    for (int64_t w = (int64_t)blockIdx.x * wpb + warp; w < W; w += (int64_t)gridDim.x * wpb) {
        cd s = cmk(0.0, 0.0);
        for (int e = lane; e < nn; e += 32) {
            cd acc = cmk(0.0, 0.0);
            for (int c = 0; c < nchunks; ++c) acc = cadd(acc, partial[(w * nchunks + c) * rec + 1 + e]);
            G[e] = acc;
            Us[e] = U[w * nn + e];
        }
        if (lane == 0) {
            for (int c = 0; c < nchunks; ++c) s = cadd(s, partial[(w * nchunks + c) * rec]);
            Sv[0] = s;
        }
        for (int e = lane; e < ne * ne; e += 32) Rs[e] = R[w * ne * ne + e];
        __syncwarp();
        // V1[k][l] = sum_{j >= ne} Gacc[j][k] conj(U[l][j])
        for (int e = lane; e < nn; e += 32) {
            int k = e / n, l = e - k * n;
            cd acc = cmk(0.0, 0.0);
            for (int j = ne; j < n; ++j) cfma(acc, G[j * n + k], cconj(Us[l * n + j]));
            V1[e] = acc;
        }
        __syncwarp();
        // Lambda[a][l] = sqrt2 Gacc[a][l] - sum_k conj(U[k][a]) V1[k][l]
        for (int e = lane; e < ne * n; e += 32) {
            int a = e / n, l = e - a * n;
            cd acc = cscale(G[a * n + l], sq2);
            for (int k = 0; k < n; ++k) cfms(acc, cconj(Us[k * n + a]), V1[k * n + l]);
            Lm[e] = acc;
        }
        __syncwarp();
        // (Lambda U_occ)[a][b] -> V1 (reused), then Mm = S U_occ^dagger + Lambda - (Lambda U_occ) U_occ^dagger
        for (int e = lane; e < ne * ne; e += 32) {
            int a = e / ne, b = e - a * ne;
            cd acc = cmk(0.0, 0.0);
            for (int k = 0; k < n; ++k) cfma(acc, Lm[a * n + k], Us[k * n + b]);
            V1[e] = acc;
        }
        __syncwarp();
        const cd S = Sv[0];
        for (int e = lane; e < ne * n; e += 32) {
            int a = e / n, l = e - a * n;
            cd acc = cadd(Lm[e], cmul(S, cconj(Us[l * n + a])));
            for (int b = 0; b < ne; ++b) cfms(acc, V1[a * ne + b], cconj(Us[l * n + b]));
            Mm[e] = acc;
        }
        // adj(R) of the upper-triangular R without divisions:
        //   N_jj = 1, N_ij = -sum_{k=i+1..j} R_ik D(i+1..k-1) N_kj,  adj_ij = D(0..i-1) D(j+1..ne-1) N_ij
        // with D(a..b) the product of the diagonal entries; one lane per column j.
        if (lane < ne) {
            const int j = lane;
            cd Ncol[QCS_MAX_N];
            for (int i = 0; i < ne; ++i) Ncol[i] = cmk(0.0, 0.0);
            Ncol[j] = cmk(1.0, 0.0);
            for (int i = j - 1; i >= 0; --i) {
                cd acc = cmk(0.0, 0.0), Dp = cmk(1.0, 0.0);
                for (int k = i + 1; k <= j; ++k) {
                    cfma(acc, cmul(Rs[i * ne + k], Dp), Ncol[k]);
                    Dp = cmul(Dp, Rs[k * ne + k]);
                }
                Ncol[i] = flip_if(acc, true);
            }
            cd post = cmk(1.0, 0.0);
            for (int k = j + 1; k < ne; ++k) post = cmul(post, Rs[k * ne + k]);
            cd pre = cmk(1.0, 0.0);
            for (int i = 0; i < ne; ++i) {
                Ad[i * ne + j] = (i <= j) ? cmul(cmul(pre, post), Ncol[i]) : cmk(0.0, 0.0);
                pre = cmul(pre, Rs[i * ne + i]);
            }
        }
        __syncwarp();
        cd ip;
        switch ((ne / 2) & 3) {
            case 0: ip = cmk(1, 0); break;
            case 1: ip = cmk(0, 1); break;
            case 2: ip = cmk(-1, 0); break;
            default: ip = cmk(0, -1); break;
        }
        const double invP = P > 0 ? 1.0 / (double)P : 0.0;
        const cd c0 = cscale(ip, 2.0 * ldexp(1.0, -(n - ne / 2)) * invP);
        // The kernel's rows are those of U_occ = U_qr W (echelon form), so the factor is
        // W^H R: adj(W^H R) = adj(R) det(conj W) W, with det(conj W) W stored in Wrot.
        const cd *Ww = Wrot + w * ((size_t)ne * ne + 1);
        cd *Ad2 = V1;  // free again
        for (int e = lane; e < ne * ne; e += 32) {
            const int a = e / ne, b = e - a * ne;
            cd acc = cmk(0.0, 0.0);
            for (int c = a; c < ne; ++c) cfma(acc, Ad[a * ne + c], Ww[c * ne + b]);
            Ad2[e] = acc;
        }
        __syncwarp();
        // grad[w][l][a] = (g^T)[a][l] = c0 sum_b adj(W^H R)[a][b] Mm[b][l]
        for (int e = lane; e < n * ne; e += 32) {
            int l = e / ne, a = e - l * ne;
            cd acc = cmk(0.0, 0.0);
            for (int b = 0; b < ne; ++b) cfma(acc, Ad2[a * ne + b], Mm[b * n + l]);
            acc = cmul(c0, acc);
            if (!cfinite(acc)) raise_status(status, QCS_ERR_NONFINITE);
            grad[w * n * ne + e] = acc;
        }
        if (lane == 0) {
            cd detR = cmk(1.0, 0.0);  // det(W^H R) = det(conj W) det R
            for (int i = 0; i < ne; ++i) detR = cmul(detR, Rs[i * ne + i]);
            overlap[w] = cmul(c0, cscale(cmul(detR, S), Ww[ne * ne].x));
        }
        __syncwarp();
    }
}

// xbar[w][g] = -sqrt_dt * i * sum_pq L[g][p][q] (Phi g^T)[q][p] / O   (sqrt_dt = 0: <v_gamma>)
__global__ void force_bias_kernel(int n, int ne, int64_t W, int nchol, const cd *__restrict__ L,
                                  const cd *__restrict__ Phi, const cd *__restrict__ ov, const cd *__restrict__ grad,
                                  double sqrt_dt, cd *__restrict__ xbar) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cd *Gf = reinterpret_cast<cd *>(smem_raw);  // Phi g^T (n x n)
    for (int64_t w = blockIdx.x; w < W; w += gridDim.x) {
        const cd *Pw = Phi + w * n * ne, *gw = grad + w * n * ne;
        for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
            int q = e / n, p = e - q * n;
            cd acc = cmk(0.0, 0.0);
            for (int j = 0; j < ne; ++j) cfma(acc, Pw[q * ne + j], gw[p * ne + j]);
            Gf[e] = acc;  // (Phi g^T)[q][p]
        }
        __syncthreads();
        const cd io = cinv(ov[w]);
        for (int g = threadIdx.x; g < nchol; g += blockDim.x) {
            const cd *Lg = L + (size_t)g * n * n;
            cd acc = cmk(0.0, 0.0);
            for (int p = 0; p < n; ++p)
                for (int q = 0; q < n; ++q) cfma(acc, Lg[p * n + q], Gf[q * n + p]);
            acc = cmul(acc, io);
            cd v = cmk(-acc.y, acc.x);  // i * tr(L G)
            xbar[w * nchol + g] = (sqrt_dt != 0.0) ? cscale(v, -sqrt_dt) : v;
        }
        __syncthreads();
    }
}

size_t grad_group_layout(GradArgs &A) {
    const int n = A.n, m = A.m, T = tri_count(m), NB = A.NB, S = m / 2;
    const size_t rows = (size_t)(n * (n + 1) > T ? n * (n + 1) : T) * sizeof(int4);
    size_t o = align16(rows);  // the walker's rows, then Y
    A.off_Q = (int)o;
    o = align16(o + rows);
    A.off_T = (int)o;
    o = align16(o + (size_t)n * ld_t(n) * sizeof(cd));
    A.off_NZ = (int)o;
    // node matrices and their entries per round, one occupied pair left to them; also B in
    // full, the assembly's limbs for any number of such pairs, the coefficients
    const int md = m - A.ne, mx = md + (A.ne > 0 ? 2 : 0), nv = NB * mx > m ? NB * mx : m;
    int nz = NB * tri_count(mx);
    if (T > nz) nz = T;
    for (int left = 0; left <= A.ne; left += 2) {
        const int need = tri_count(md + left) + 2 * (md + left) * (A.ne - left);
        if (need > nz) nz = need;
    }
    if (m * n > nz) nz = m * n;
    A.nz = nz;
    A.nv = nv;
    o = align16(o + nz * sizeof(cd));
    A.off_g = (int)o;  // Gauss vectors; the four vectors of grad_full_nodes
    o = align16(o + (size_t)(nv > 2 * m ? nv : 2 * m) * sizeof(FxGauss));
    A.off_pv = (int)o;
    o = align16(o + (size_t)(A.ne / 2 + nv / 2) * sizeof(fx2));
    A.off_pe = (int)o;
    o = align16(o + (size_t)(A.ne / 2 + nv / 2) * sizeof(int));
    A.off_se = (int)o;
    o = align16(o + (size_t)(m + nv) * sizeof(int));
    A.off_perm = (int)o;
    o = align16(o + (size_t)m + 3 * nv);
    A.off_cf = (int)o;
    o = align16(o + (size_t)kMaxNBG * sizeof(cd));
    A.off_invh = (int)o;
    o = align16(o + (size_t)S * sizeof(cd));
    A.off_hist = (int)o;
    o = align16(o + (size_t)(S + 1) * m + 2 * S);
    A.off_scr = (int)o;
    o = align16(o + sizeof(GradShared));
    return o;
}

}  // namespace

qcs_status qcs_launch_grad(qcs_ctx *ctx, const qcs_grad_launch &L, cudaStream_t st) {
    GradArgs A;
    memset(&A, 0, sizeof(A));
    A.n = L.n;
    A.ne = L.ne;
    A.m = 2 * L.n - L.ne;
    A.d = L.n - L.ne;
    A.nev = L.plan.nev;
    A.all = L.plan.all;
    A.chunk = L.chunk;
    A.nchunks = L.nchunks;
    A.W = L.W;
    A.P = L.P;
    A.tab_bytes = (int)align16((size_t)tri_count(A.m) * sizeof(uint16_t));
    A.Ut = L.Ut;
    A.Qh = L.s->Qh;
    A.idx = L.s->idx;
    A.d_count = L.s->d_count;
    A.partial = L.partial;
    A.counter = L.counter;
    A.status = ctx->d_status;
    fx_make_plan(L.plan, A.plan);
    for (int k = 0; k < L.plan.nev; ++k) {
        A.wnode[k] = L.plan.wnode[k];
        A.gamma[k] = L.plan.gamma[k];
    }
    // Node matrices per round (NB) and groups per block: the most resident groups
    // (at most 8 per SM, i.e. four warps per SM sub-partition), then the largest NB.
    int best_nb = 0, best_g = 1, best_score = -1;
    const int nbmax = L.plan.nev < kMaxNBG ? L.plan.nev : kMaxNBG;
    for (int nb = nbmax; nb >= 1; --nb) {
        A.NB = nb;
        const size_t gb = grad_group_layout(A);
        for (int g = 2; g >= 1; --g) {
            const size_t sm = (size_t)A.tab_bytes + (size_t)g * gb;
            if (sm > ctx->smem_optin) continue;
            int per_sm = (int)(ctx->smem_per_sm / (sm + 1024));
            if (per_sm > 4) per_sm = 4;
            int groups = per_sm * g;
            if (groups > 8) groups = 8;
            const int score = groups * 16 + nb;
            if (per_sm >= 1 && score > best_score) {
                best_score = score;
                best_nb = nb;
                best_g = g;
            }
        }
    }
    if (best_nb == 0) return qcs_fail(ctx, QCS_ERR_UNSUPPORTED, "grad kernel: shared memory too large");
    A.NB = best_nb;
    A.group_bytes = (int)grad_group_layout(A);
    const int threads = best_g * kGroup;
    size_t smem = (size_t)A.tab_bytes + (size_t)best_g * A.group_bytes;
    if (qcs_set_smem(ctx, (const void *)grad_pair_kernel, smem) != QCS_OK) return QCS_ERR_CUDA;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, grad_pair_kernel, threads, smem) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    int64_t ntiles = L.W * L.nchunks;
    int64_t blocks = (int64_t)ctx->num_sms * per_sm;
    int64_t need = (ntiles + best_g - 1) / best_g;
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    if (cudaMemsetAsync(L.counter, 0, sizeof(unsigned long long), st) != cudaSuccess)
        return qcs_fail(ctx, QCS_ERR_CUDA, "grad tile counter reset");
    qcs_prof_begin(ctx, st);
    grad_pair_kernel<<<(unsigned)blocks, threads, smem, st>>>(A);
    qcs_prof_end(ctx, st);
    qcs_status r = qcs_check_launch(ctx, "grad_pair_kernel");
    if (r != QCS_OK) return r;
    const int n = L.n, ne = L.ne;
    const int ewpb = 4;
    size_t esm = (size_t)ewpb * (4 * n * n + 2 * ne * n + 2 * ne * ne + 2) * sizeof(cd);
    if (qcs_set_smem(ctx, (const void *)grad_epilogue_kernel, esm) != QCS_OK) return QCS_ERR_CUDA;
    int64_t eb = (L.W + ewpb - 1) / ewpb;
    if (eb > (int64_t)ctx->num_sms * 8) eb = (int64_t)ctx->num_sms * 8;
    grad_epilogue_kernel<<<(unsigned)eb, ewpb * 32, esm, st>>>(n, ne, L.W, L.P, L.nchunks, L.partial, L.U, L.R, L.Wrot,
                                                               L.overlap, L.grad, ctx->d_status);
    return qcs_check_launch(ctx, "grad_epilogue_kernel");
}

qcs_status qcs_launch_force_bias(qcs_ctx *ctx, int n, int ne, int64_t W, int nchol, const cd *L, const cd *walkers,
                                 const cd *overlap, const cd *grad, double sqrt_dt, cd *xbar, cudaStream_t st) {
    if (W == 0 || nchol == 0) return QCS_OK;
    size_t smem = (size_t)n * n * sizeof(cd);
    int64_t blocks = W < (int64_t)ctx->num_sms * 8 ? W : (int64_t)ctx->num_sms * 8;
    force_bias_kernel<<<(unsigned)blocks, 128, smem, st>>>(n, ne, W, nchol, L, walkers, overlap, grad, sqrt_dt, xbar);
    return qcs_check_launch(ctx, "force_bias_kernel");
}
