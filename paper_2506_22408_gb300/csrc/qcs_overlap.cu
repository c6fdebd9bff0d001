// qcs_overlap.cu -- walker x snapshot shadow overlaps without a tensor-core congruence.
//
// For a pair (walker w, snapshot p) the estimator of Sec. "Classical shadows
// and the evaluation of overlaps" needs the coefficients of
// pf(A(z)), A(z) = C_0^(s) + z B^(s)  (Eqs. a_mat, b_mat).  The kernel forms, all in fixed
// point on the integer pipe (qcs_fixed.cuh, qcs_fxcong.cuh: the FP64 pipe, one 32-lane FMA
// per 76 clocks and scheduler, bound it before):
//
//  1. T = Ut Qt^T (n x 2n complex): Ut holds the walker's orbitals (rows of
//     U^T, occupied rows / sqrt2), Qt the snapshot's complexified sign-folded
//     rows.  Row j of T is the selected row of W^* M_phi Q'^T for an occupied
//     mode j; for an empty mode the two selected real rows are (Re T_j, -Im T_j).
//     The walker prep leaves the orbitals in echelon form, so T skips the exact
//     zeros of Ut.  Signed permutations gather T from Ut.
//  2. B^(s)_ab = sum_k X_a,2k X_b,2k+1 - X_a,2k+1 X_b,2k  (X = selected rows),
//     i.e. X J X^T with J the canonical skew form (C_b was folded into Qt).  Above 16
//     modes K = Ut [H1 | G2] takes the place of T and B^(s) follows from K by n-term sums.
//  3. pf(B + w_k D) at the node plan's evaluation points w_k (a Gauss rule on the
//     unit circle by default, roots of unity on request), D = C_0^(s): the node
//     matrices differ only in their empty x empty block, so the occupied block is
//     eliminated once (pivots inside that block) and each node's 2d x 2d complement
//     is eliminated by Parlett-Reid with partial pivoting, the nodes in lockstep.
//  4. S_p = sum_k gamma_k pf_k, where gamma_k folds the node plan's weights, the
//     inverse-channel weights C(2n,2x)/C(n,x) and the palindromic symmetry
//     c_{n-x} = c_x of parity +1 snapshots (parity -1 snapshots are exactly zero
//     and skipped).
//
// Tiles are (walker, chunk of snapshots) owned by a block of four warps; each warp
// (n <= 16) or each pair of warps (n > 16, 64-thread groups) takes every
// snapshot of the tile in turn and writes one partial sum per warp slot, reduced
// in a fixed order afterwards, so the result does not depend on scheduling.
#include "qcs_internal.h"
#include "qcs_fxcong.cuh"
#include "qcs_pairfp64.cuh"

namespace {


struct PairArgs {
    int n, ne, m, NB, all, chunk, nchunks;
    int grp;          // n > 16: two warps share a pair
    int64_t W, P;
    int team_bytes;   // shared bytes per team (one warp, or two)
    int tab_bytes;    // shared bytes of the pair table (per block)
    int ut_bytes;     // shared bytes of the walker rows Ut (per block)
    int off_T, off_U, off_pv, off_scr, npv;  // byte offsets in a team's region (staged rows, then B^(s), at 0)
    const cd *Ut;
    const cd *pref;
    const cd *Qt;
    const cd *Qh;        // rows [H1^T; G2^T] of the dense snapshots (null: T and B from Qt)
    const uint8_t *gth;  // gather codes of signed-permutation snapshots (or null)
    const int *idx;
    const int *d_count;
    cd *partial;
    cd *per_pair;
    unsigned *status;
    FxPlan plan;
};

// What a team's warps exchange.
struct PairScratch {
    unsigned red[4];
    cd part;
    int8_t rs[2 * QCS_MAX_N];  // row scales of the pair's snapshot
};

// The sum over the pairs of walker w with the snapshots p0, p0 + teams, ... below p1 of the list, on
// the team's first thread.  Guarded pairs whose pivots show lost bits are evaluated in FP64.
template <int NW, bool kGuarded>
__device__ __forceinline__ cd tile_pairs(const PairArgs &A, int64_t w, int64_t p0, int64_t p1, int teams, int fU,
                                         unsigned char *tb, const int4 *Us, const uint16_t *tab, int bar, int wid,
                                         int lane) {
    const int n = A.n, n2 = 2 * n;
    int4 *Qs = reinterpret_cast<int4 *>(tb);            // half of the snapshot's rows
    fx2 *Xs = reinterpret_cast<fx2 *>(tb);              // B^(s), once T is formed
    int4 *Ts = reinterpret_cast<int4 *>(tb + A.off_T);
    fx2 *Ns = reinterpret_cast<fx2 *>(tb + A.off_T);    // node matrices, once B^(s) is formed
    fx2 *pv = reinterpret_cast<fx2 *>(tb + A.off_pv);
    PairScratch *scr = reinterpret_cast<PairScratch *>(tb + A.off_scr);
    const FxWork wk = {reinterpret_cast<FxGauss *>(tb + A.off_U), pv, reinterpret_cast<int *>(pv + A.npv + A.ne / 2),
                       A.npv};
    const FxTeam<NW> tm = {32 * wid + lane, lane, wid, bar, scr->red};
    cd acc = cmk(0.0, 0.0);
    for (int64_t pq = p0; pq < p1; pq += teams) {
        const int64_t q = A.all ? pq : (int64_t)A.idx[pq];
        if (!QCS_IN_BOUNDS(q >= 0 && q < A.P, A.status)) continue;  // team-uniform
        const uint8_t *gq = A.gth ? A.gth + q * n2 : nullptr;
        const bool gat = gq && gq[0] != 0xFF, fromK = !gat && A.Qh;
        cd S = cmk(__longlong_as_double(0x7ff8000000000000ll), 0.0);
        bool finite = true;
        int fT = fU, par = 0;
        tm.sync();  // the previous pair is done with the team's region
        if (gat) {
            fx_gather_T(n, Us, gq, Ts, tm.t, tm.NT);  // signed permutation: no products
            fT = fU - 1;
        } else {
            // T (or K) by column halves: half of the snapshot's rows staged at a time
            const cd *Qr = (A.Qh ? A.Qh : A.Qt) + q * n2 * n;
            const unsigned key = fromK ? fx_max_key(Qr, n2 * n, lane) : fx_balance_rows(n, Qr, scr->rs, lane);
            finite = key < 0x7ff00000u;
            const int fQ = fx_fraction(key, 57);
            unsigned top = 0u;
            tm.sync();
            for (int h = 0; h < 2 && finite; ++h) {
                fx_stage_rows(n, n * n, Qr + (int64_t)h * n * n, fQ, fromK ? nullptr : scr->rs + h * n, Qs, tm.t, tm.NT);
                tm.sync();
                top |= fx_build_T(n, A.ne, Us, Qs, reinterpret_cast<fx2 *>(Ts), h * n, tm.t, tm.NT);
                tm.sync();
            }
            if (finite) {
                top = tm.or_put(top, par);
                tm.sync();
                const int b = fx_top_bits(tm.or_get(top, par));
                par ^= 1;
                fT = fU + fQ - 58 + 56 - b;
                if (fromK) fx_T_limbs<kFxS>(n, Ts, b, tm.t, tm.NT);
                else fx_T_limbs<kFxST>(n, Ts, b, tm.t, tm.NT);
            }
        }
        tm.sync();
        if (finite) {
            bool shared = true, ok, lost = false;
#pragma unroll 1
            do {  // rarely a second time: B^(s) again, every node matrix in full
                unsigned top = fromK ? fx_build_B_from_K(n, A.ne, Us, Ts, Xs, tab, tm.t, tm.NT)
                                     : fx_build_B(n, A.ne, Ts, Xs, tab, tm.t, tm.NT);
                top = tm.or_put(top, par);
                tm.sync();
                const int mb = fx_top_bits(tm.or_get(top, par));
                par ^= 1;
                tm.sync();  // the words of the reduction are free again
                S = fx_pair_eliminate<kGuarded>(tm, A.m, A.ne, shared, A.NB, A.plan, wk, Xs, Ns,
                                                fromK ? fT + fU - 58 : 2 * fT - 56, mb, tab, ok, &lost);
                shared = false;
                tm.sync();
            } while (!ok && !lost);
            if (kGuarded && lost) {  // in FP64, the first warp's value alone
                S = fp64_pair_sum(tm, n, A.ne, A.plan, A.Ut + w * n * n, A.Qt + q * n2 * n, gat ? gq : nullptr,
                                  reinterpret_cast<cd *>(Xs), reinterpret_cast<cd *>(Ns),
                                  reinterpret_cast<cd *>(wk.GV), tab);
                if (wid != 0) S = cmk(0.0, 0.0);
            }
        }
        if (NW > 1) {  // the other warp's nodes
            if (wid == 1 && lane == 0) scr->part = finite ? S : cmk(0.0, 0.0);
            tm.sync();
            if (wid == 0 && lane == 0) S = cadd(S, scr->part);
        }
        if (tm.t == 0) {
            if (!cfinite(S)) raise_status(A.status, QCS_ERR_NONFINITE);
            acc = cadd(acc, S);
            if (A.per_pair) A.per_pair[w * A.P + q] = cmul(A.pref[w], S);
        }
    }
    return acc;
}
// One tile of system A: walker w = tile / nchunks, the tile's snapshots spread over the
// block's teams of NW warps; each team writes one partial sum, in its first warp's slot (zero
// in the second's).  Every thread of the block calls this (it contains block barriers
// around the shared walker rows).  Returns whether the tile was left to the other pass.
//
// Guarded are the tiles in which B^(s) can hold entries of very different sizes, of which one
// scale loses the small ones: a walker that has such entries where the set has signed
// permutations, which copy them (the exact zeros of a basis determinant stay exact), and all
// tiles of a set with a dense snapshot that is sparse or graded itself; both counted when the
// set is built.  Haar-random snapshots mix the entries.  The guarded tiles are a pass of their
// own, a call after the loop over the others: with the guard and the FP64 call in the only loop,
// 12 modes took 13.88 instead of 13.26 ms and 8 modes 152 instead of 138 us without a single
// guarded pair; with the choice made for each pair 13.45 ms and 143 us, for each tile 13.35 ms
// and 141 us.
template <int NW, bool kGuarded>
__device__ bool run_tile(const PairArgs &A, int64_t tile, int64_t L, unsigned char *base, int4 *Us,
                         const uint16_t *tab, int warp, int wpb, int lane) {
    const int n = A.n;
    const int team = warp / NW, wid = warp % NW, teams = wpb / NW;
    const int span = A.chunk * wpb;  // snapshots per tile; team g takes every teams-th
    // chunk-major tile order: consecutive tiles share one snapshot chunk and run over
    // the walkers (whose rows all fit in L2), so each snapshot is fetched from HBM once
    const int ch = (int)(tile / A.W);
    const int64_t w = tile - (int64_t)ch * A.W;
    const int64_t p0 = (int64_t)ch * span;
    const int64_t p1 = p0 + span < L ? p0 + span : L;
    // the tile from the queue and the parity +1 count address this system's buffers
    // (block-uniform: every thread leaves before the first barrier)
    if (!QCS_IN_BOUNDS(tile >= 0 && ch < A.nchunks && L >= 0 && L <= A.P, A.status)) return false;
    __syncthreads();  // previous tile's readers of Us are done
    int fU = 0;
    if (p0 < L) {
        const cd *Utw = A.Ut + w * n * n;
        const unsigned key = fx_max_key(Utw, n * n, lane);
        fU = fx_fraction(key, 57);
        const bool guard = A.d_count[2] > 0 || (A.d_count[1] > 0 && fx_wide(Utw, n * n, key, lane));
        if (guard != kGuarded) return true;  // block-uniform
        fx_stage_rows(n, n * n, Utw, fU, nullptr, Us, threadIdx.x, blockDim.x);
    } else if (kGuarded) {
        return true;
    }
    __syncthreads();
    cd acc = cmk(0.0, 0.0);
    if (p0 < L)
        acc = tile_pairs<NW, kGuarded>(A, w, p0 + team, p1, teams, fU, base + (size_t)team * A.team_bytes, Us, tab,
                                       1 + team, wid, lane);
    if (lane == 0) A.partial[(w * A.nchunks + ch) * wpb + warp] = wid == 0 ? acc : cmk(0.0, 0.0);
    return false;
}

// One or several systems (different n, ne, walkers, snapshots) in one persistent
// launch.  Blocks pull tiles from a global counter (no fixed stride, so no block
// can be dealt only empty tiles); the tile space lists the systems in decreasing
// cost per tile, so the largest tiles are handed out first and the small ones
// fill the tail.
struct BatchArgs {
    int nsys;
    int tab_bytes, ut_bytes, work_bytes;  // maxima over the systems
    int max_m;
    int64_t tile_end[QCS_MAX_SYSTEMS];    // cumulative tile counts in queue order
    unsigned long long *counter;          // tiles handed out in the first pass and in the second
    PairArgs sys[QCS_MAX_SYSTEMS];         // in queue order
};

// The guarded tiles, or the others; whether this block met tiles of the other kind.
template <int NWS, bool kGuarded>
__device__ __forceinline__ bool overlap_tiles(const BatchArgs &B, unsigned char *smem_raw, long long *next_tile) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    const uint16_t *tab = reinterpret_cast<uint16_t *>(smem_raw);
    int4 *Us = reinterpret_cast<int4 *>(smem_raw + B.tab_bytes);
    unsigned char *base = smem_raw + B.tab_bytes + B.ut_bytes;
    const int64_t total = B.tile_end[B.nsys - 1];
    bool other = false;
    for (;;) {
        __syncthreads();  // every thread has read the previous tile index
        if (threadIdx.x == 0) *next_tile = (long long)atomicAdd(B.counter + (kGuarded ? 1 : 0), 1ull);
        __syncthreads();
        const int64_t t = *next_tile;
        if (t >= total) break;
        int s = 0;
        while (t >= B.tile_end[s]) ++s;
        const int64_t local = t - (s > 0 ? B.tile_end[s - 1] : 0);
        const PairArgs &A = B.sys[s];
        const int64_t L = A.all ? A.P : (int64_t)(*A.d_count);
        if ((NWS & 2) && (!(NWS & 1) || A.grp))
            other |= run_tile<2, kGuarded>(A, local, L, base, Us, tab, warp, wpb, lane);
        else other |= run_tile<1, kGuarded>(A, local, L, base, Us, tab, warp, wpb, lane);
    }
    return other;
}
template <int NWS>
static __device__ __noinline__ void guarded_tiles(const BatchArgs &B, unsigned char *smem_raw, long long *next_tile) {
    overlap_tiles<NWS, true>(B, smem_raw, next_tile);
}

// NWS: bit 0 set when a system of the launch runs one warp per pair, bit 1 when one runs two;
// a kind that does not occur is left out of the kernel (its instructions and registers).
template <int NWS>
__global__ void __launch_bounds__(128, 4) pair_overlap_kernel(const __grid_constant__ BatchArgs B) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ long long next_tile;
    // the pair table, the walker rows and the teams' workspaces fit the launch's shared memory
    if (!QCS_IN_BOUNDS(tri_count(B.max_m) * (int)sizeof(uint16_t) <= B.tab_bytes &&
                           (size_t)B.tab_bytes + B.ut_bytes + B.work_bytes <= dyn_smem_bytes(),
                       B.sys[0].status))
        return;
    build_pair_table(reinterpret_cast<uint16_t *>(smem_raw), tri_count(B.max_m));
    // a block that met guarded tiles takes part in the second pass, over all tiles
    if (overlap_tiles<NWS, false>(B, smem_raw, &next_tile)) guarded_tiles<NWS>(B, smem_raw, &next_tile);
}

// One warp per walker: lanes sum strided partials, then a fixed-order tree.
__global__ void reduce_kernel(int64_t W, int64_t P, int nparts, const cd *__restrict__ partial,
                              const cd *__restrict__ pref, cd *__restrict__ overlap) {
    int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= W) return;
    cd s = cmk(0.0, 0.0);
    for (int c = lane; c < nparts; c += 32) s = cadd(s, partial[w * nparts + c]);
    s = warp_csum(s);
    if (lane != 0) return;
    double inv = P > 0 ? 1.0 / (double)P : 0.0;
    overlap[w] = cscale(cmul(pref[w], s), inv);
}

}  // namespace

namespace {

// Shared workspace of one team for nb node matrices per round; returns its bytes.  The first
// region holds half of the snapshot's rows, then B^(s); the second T (or K), then the node
// matrices: NB complements of 2d x 2d, or one full matrix.
size_t pair_team_layout(PairArgs &A, int NB) {
    const int n = A.n, m = A.m, T = tri_count(m), d2 = m - A.ne, Tn = tri_count(d2);
    const int vm = m > NB * d2 ? m : NB * d2;
    const auto most = [](int a, int b) { return a > b ? a : b; };
    size_t o = (size_t)most(n * (n + 1), T) * sizeof(int4);
    A.off_T = (int)o;
    o += (size_t)most(most(n * ld_t(n), T), NB * Tn) * sizeof(int4);
    A.off_U = (int)o;
    o += (size_t)vm * sizeof(FxGauss);
    A.off_pv = (int)o;
    A.npv = pv_records(vm, NB);
    o = align16(o + pv_bytes(vm, NB, A.ne));
    A.off_scr = (int)o;
    return align16(o + sizeof(PairScratch));
}

}  // namespace

int qcs_pair_warps_per_block() { return 4; }

bool qcs_pair_forms_K(int n, int config) { return n > 16 && qcs_decode_config(config).warps != 1; }

namespace {

// Fill the per-system arguments and shared layout of one pair launch.
void setup_pair_args(qcs_ctx *ctx, const qcs_pair_launch &L, PairArgs &A) {
    memset(&A, 0, sizeof(A));
    A.n = L.n;
    A.ne = L.ne;
    A.m = 2 * L.n - L.ne;
    A.all = L.plan.all;
    A.chunk = L.chunk;
    A.nchunks = L.nchunks;
    A.W = L.W;
    A.P = L.P;
    const qcs_config cfg = qcs_decode_config(L.config);
    A.grp = qcs_pair_forms_K(L.n, L.config);  // n > 16: two warps per pair unless one is configured
    const int n = A.n, m = A.m, T = tri_count(m), nev = L.plan.nev;
    const int teams = qcs_pair_warps_per_block() / (A.grp ? 2 : 1);
    A.tab_bytes = (int)align16((size_t)T * sizeof(uint16_t));
    A.ut_bytes = (int)align16((size_t)n * (n + 1) * sizeof(int4));
    const auto block = [&](int nb) { return (size_t)A.tab_bytes + A.ut_bytes + teams * pair_team_layout(A, nb) + 1024; };
    // Node matrices per round: the requested count, or by default the largest balanced one
    // (at most kMaxNB) that costs no resident block: more nodes share a round's pivot work,
    // but warps in flight hide the eliminations' latencies.
    int NB = 1;
    const auto resident = [&](int nb) {
        const int b = (int)((ctx->smem_optin + 1024) / block(nb));
        return b < 4 ? b : 4;
    };
    if (cfg.nb > 0) {
        NB = cfg.nb < nev ? cfg.nb : nev;
        if (NB > kMaxNB) NB = kMaxNB;
        while (NB > 1 && block(NB) > ctx->smem_optin) --NB;
    } else {
        for (int rounds = 1; rounds <= nev; ++rounds) {
            const int nb = (nev + rounds - 1) / rounds;
            if (nb <= kMaxNB && resident(nb) >= 1 && resident(nb) >= resident(1)) {
                NB = nb;
                break;
            }
        }
    }
    A.NB = NB;
    A.team_bytes = (int)pair_team_layout(A, NB);
    A.Ut = L.Ut;
    A.pref = L.pref;
    A.Qt = L.s->Qt;
    A.Qh = A.grp ? L.s->Qh : nullptr;  // two warps form K and B from K; one T
    A.gth = L.s->gth;
    A.idx = L.s->idx;
    A.d_count = L.s->d_count;
    A.partial = L.partial;
    A.per_pair = L.per_pair;
    A.status = ctx->d_status;
    fx_make_plan(L.plan, A.plan);
}

}  // namespace

qcs_status qcs_launch_pairs(qcs_ctx *ctx, const qcs_pair_launch &L, cudaStream_t st) {
    return qcs_launch_pairs_batched(ctx, 1, &L, L.counter, st);
}

qcs_status qcs_launch_pairs_batched(qcs_ctx *ctx, int nsys, const qcs_pair_launch *Ls, unsigned long long *counter,
                                    cudaStream_t st) {
    if (nsys < 1 || nsys > QCS_MAX_SYSTEMS) return QCS_ERR_ARG;
    BatchArgs B;
    memset(&B, 0, sizeof(B));
    B.nsys = nsys;
    B.counter = counter;
    // queue order: decreasing estimated cost of one tile
    int order[QCS_MAX_SYSTEMS];
    double cost[QCS_MAX_SYSTEMS];
    for (int i = 0; i < nsys; ++i) {
        order[i] = i;
        cost[i] = qcs_overlap_flops_nev(Ls[i].n, Ls[i].ne, Ls[i].plan.nev, true) *
                  (double)Ls[i].chunk;
    }
    for (int i = 0; i < nsys; ++i)
        for (int j = i + 1; j < nsys; ++j)
            if (cost[order[j]] > cost[order[i]]) {
                int t = order[i];
                order[i] = order[j];
                order[j] = t;
            }
    int64_t acc = 0;
    for (int q = 0; q < nsys; ++q) {
        const qcs_pair_launch &L = Ls[order[q]];
        setup_pair_args(ctx, L, B.sys[q]);
        acc += L.W * L.nchunks;
        B.tile_end[q] = acc;
        if (B.sys[q].tab_bytes > B.tab_bytes) B.tab_bytes = B.sys[q].tab_bytes;
        if (B.sys[q].ut_bytes > B.ut_bytes) B.ut_bytes = B.sys[q].ut_bytes;
        const int work = B.sys[q].team_bytes * (qcs_pair_warps_per_block() / (B.sys[q].grp ? 2 : 1));
        if (work > B.work_bytes) B.work_bytes = work;
        if (B.sys[q].m > B.max_m) B.max_m = B.sys[q].m;
    }
    if (acc == 0) return QCS_OK;
    const int wpb = qcs_pair_warps_per_block();
    size_t smem = (size_t)B.tab_bytes + B.ut_bytes + B.work_bytes;
    if (smem + 64 > ctx->smem_optin)  // + the kernel's static tile index
        return qcs_fail(ctx, QCS_ERR_UNSUPPORTED, "batched kernel: shared memory too large");
    int kinds = 0;
    for (int q = 0; q < nsys; ++q) kinds |= B.sys[q].grp ? 2 : 1;
    void (*const kern)(BatchArgs) = kinds == 1 ? pair_overlap_kernel<1> : kinds == 2 ? pair_overlap_kernel<2> : pair_overlap_kernel<3>;
    const void *kfn = (const void *)kern;
    if (qcs_set_smem(ctx, kfn, smem) != QCS_OK) return QCS_ERR_CUDA;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, wpb * 32, smem) !=
            cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    int64_t blocks = (int64_t)ctx->num_sms * per_sm;
    if (blocks > acc) blocks = acc;
    cudaError_t e = cudaMemsetAsync(counter, 0, 2 * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return qcs_fail(ctx, QCS_ERR_CUDA, "batched counter reset");
    qcs_prof_begin(ctx, st);
    kern<<<(unsigned)blocks, wpb * 32, smem, st>>>(B);
    qcs_prof_end(ctx, st);
    return qcs_check_launch(ctx, "pair_overlap_kernel");
}

qcs_status qcs_launch_reduce(qcs_ctx *ctx, int64_t W, int64_t P, int nparts, const cd *partial, const cd *pref,
                             cd *overlap, cudaStream_t st) {
    if (W == 0) return QCS_OK;
    int64_t blocks = (W * 32 + 127) / 128;
    reduce_kernel<<<(unsigned)blocks, 128, 0, st>>>(W, P, nparts, partial, pref, overlap);
    return qcs_check_launch(ctx, "reduce_kernel");
}
