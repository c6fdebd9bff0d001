// qcs_pfaff.cu -- Pfaffian sums of pairs whose covariance another kernel has formed.
//
// The tensor-core congruence (qcs_tcpair.cu) leaves B^(s) of a batch of pairs in device
// memory as fixed point (qcs_fixed.cuh: packed triangle, the empty modes' rows first, then
// its fraction bits); pfaffian_kernel takes one pair per warp, copies the record into
// shared memory and evaluates sum_k gamma_k pf(B + w_k D), one value per pair;
// pair_sum_kernel adds a walker's values in snapshot order.
//
// Why two kernels: the operands of the congruence take 72 KB of shared memory per four
// warps, so a fused kernel holds 12 warps per SM, and the eliminations, chains of
// dependent integer instructions with 11 KB per warp, then leave half of the issue slots
// empty (ncu: 51 % at 3 warps per scheduler).  On their own they run with 20 warps per SM.
// The records cost 2 x 16 (tri(m) + 1) bytes of memory traffic per pair (8.8 KB at n = 16,
// ne = 8).
#include "qcs_fixed.cuh"
#include "qcs_internal.h"

namespace {

constexpr int kPfWarps = 4;  // warps per block

struct PfArgs {
    int m, ne, NB;
    int64_t W;       // walkers of the batch
    int64_t P;       // snapshots of the set
    int64_t p0;      // first list position of the batch
    int span;        // list positions of the batch, at most
    int rec_bytes;   // bytes per record
    int ws_bytes;    // shared workspace per warp
    int off_N, off_U, off_pv, npv;  // byte offsets in it (B^(s) at 0); off_N after a full B
    const unsigned char *rec;
    const int *d_count;
    const int *idx;
    const cd *pref;
    cd *sum;         // W x span
    cd *per_pair;    // W x P or null
    unsigned *status;
    FxPlan plan;
};

__global__ void __launch_bounds__(32 * kPfWarps, 5) pfaffian_kernel(const __grid_constant__ PfArgs A) {
    extern __shared__ __align__(16) unsigned char smem_pf[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int T = tri_count(A.m), Tn = tri_count(A.m - A.ne);
    const int tab_bytes = (int)align16((size_t)T * sizeof(uint16_t));
    if (!QCS_IN_BOUNDS(tab_bytes + kPfWarps * A.ws_bytes <= (int)dyn_smem_bytes(), A.status)) return;
    uint16_t *tab = reinterpret_cast<uint16_t *>(smem_pf);
    build_pair_table(tab, T);
    __syncthreads();
    unsigned char *ws = smem_pf + tab_bytes + (size_t)warp * A.ws_bytes;
    fx2 *X = reinterpret_cast<fx2 *>(ws);
    fx2 *pv = reinterpret_cast<fx2 *>(ws + A.off_pv);
    const FxWork wk = {reinterpret_cast<FxGauss *>(ws + A.off_U), pv,
                       reinterpret_cast<int *>(pv + A.npv + A.ne / 2), A.npv};
    const FxWarp tm = {lane, lane, 0, 0, nullptr};
    const int64_t L = *A.d_count;
    const int64_t live = L - A.p0 < 0 ? 0 : (L - A.p0 < A.span ? L - A.p0 : A.span);
    const unsigned items = (unsigned)(live * A.W), step = gridDim.x * kPfWarps;
    for (unsigned i = blockIdx.x * kPfWarps + warp; i < items; i += step) {
        const unsigned p = i / (unsigned)A.W, w = i - p * (unsigned)A.W;
        const unsigned char *rec = A.rec + (size_t)i * A.rec_bytes;
        const int2 h = *reinterpret_cast<const int2 *>(rec + (size_t)T * sizeof(fx2));
        bool shared = true, ok;
        cd S;
#pragma unroll 1
        do {  // rarely a second time: B^(s) again, every node matrix in full
            const fx2 *src = reinterpret_cast<const fx2 *>(rec);
            for (int e = lane; e < T; e += 32) X[e] = src[e];
            __syncwarp();
            // the node matrices follow S, or B^(s)
            S = fx_pair_eliminate(tm, A.m, A.ne, shared, A.NB, A.plan, wk, X,
                                  shared ? X + Tn : reinterpret_cast<fx2 *>(ws + A.off_N), h.x, h.y, tab, ok);
            shared = false;
            __syncwarp();
        } while (!ok);
        if (lane == 0) {
            if (!cfinite(S)) raise_status(A.status, QCS_ERR_NONFINITE);
            A.sum[(size_t)w * A.span + p] = S;
            if (A.per_pair) {
                const int64_t q = A.idx[A.p0 + p];
                if (QCS_IN_BOUNDS(q >= 0 && q < A.P, A.status)) A.per_pair[w * A.P + q] = cmul(A.pref[w], S);
            }
        }
        __syncwarp();
    }
}

// partial[w][c] = sum over the batch's list positions of a walker's values, in a fixed
// order (a warp per walker: strided lane sums, then a tree).
__global__ void pair_sum_kernel(int64_t W, int64_t p0, int span, const int *__restrict__ d_count,
                                const cd *__restrict__ sum, cd *__restrict__ partial, int nchunks) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= W) return;
    const int64_t L = *d_count;
    const int64_t live = L - p0 < 0 ? 0 : (L - p0 < span ? L - p0 : span);
    cd s = cmk(0.0, 0.0);
    for (int p = lane; p < live; p += 32) s = cadd(s, sum[(size_t)w * span + p]);
    s = warp_csum(s);
    if (lane == 0) partial[w * nchunks] = s;
}

// Shared workspace of one warp for NB complements per round: B^(s) (later S and after it
// the node matrices; a second full triangle for the full eliminations), the Gauss vectors
// and the records; returns its bytes.
size_t pf_layout(PfArgs &A, int NB) {
    const int m = A.m, T = tri_count(m), d2 = m - A.ne, Tn = tri_count(d2);
    const int vm = m > NB * d2 ? m : NB * d2;
    const size_t mats = (size_t)(2 * T > (NB + 1) * Tn ? 2 * T : (NB + 1) * Tn) * sizeof(fx2);
    A.off_N = T * (int)sizeof(fx2);
    size_t o = align16(mats);
    A.off_U = (int)o;
    o = align16(o + (size_t)vm * sizeof(FxGauss));
    A.off_pv = (int)o;
    A.npv = pv_records(vm, NB);
    return align16(o + pv_bytes(vm, NB, A.ne));
}

}  // namespace

int qcs_pf_rec_bytes(int n, int ne) { return (tri_count(2 * n - ne) + 1) * (int)sizeof(fx2); }

qcs_status qcs_launch_pfaffians(qcs_ctx *ctx, const qcs_pf_launch &L, cudaStream_t st) {
    PfArgs A;
    memset(&A, 0, sizeof(A));
    A.m = 2 * L.n - L.ne;
    A.ne = L.ne;
    const int nev = L.plan->nev;
    A.W = L.W;
    A.P = L.s->P;
    A.p0 = L.p0;
    A.span = L.span;
    A.rec_bytes = qcs_pf_rec_bytes(L.n, L.ne);
    A.rec = L.rec;
    A.d_count = L.s->d_count;
    A.idx = L.s->idx;
    A.pref = L.pref;
    A.sum = L.sum;
    A.per_pair = L.per_pair;
    A.status = ctx->d_status;
    fx_make_plan(*L.plan, A.plan);
    // node matrices per round: the requested count, or the largest balanced one that leaves
    // 16 warps per SM
    const size_t tab = align16((size_t)tri_count(A.m) * sizeof(uint16_t));
    const auto block = [&](int nb) { return tab + kPfWarps * pf_layout(A, nb); };
    int NB = 1;
    const int want = qcs_decode_config(L.config).nb;
    if (want > 0) {
        NB = want < nev ? want : nev;
        if (NB > kMaxNB) NB = kMaxNB;
        while (NB > 1 && block(NB) > ctx->smem_optin) --NB;
    } else {
        for (int rounds = 1; rounds <= nev; ++rounds) {
            const int nb = (nev + rounds - 1) / rounds;
            if (nb <= kMaxNB && 4 * (block(nb) + 1024) <= ctx->smem_per_sm) {
                NB = nb;
                break;
            }
        }
    }
    A.NB = NB;
    const size_t smem = block(NB);
    A.ws_bytes = (int)pf_layout(A, NB);
    const void *fn = (const void *)pfaffian_kernel;
    if (qcs_set_smem(ctx, fn, smem) != QCS_OK) return QCS_ERR_CUDA;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * kPfWarps, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    int64_t blocks = (int64_t)ctx->num_sms * per_sm;
    const int64_t need = (A.W * A.span + kPfWarps - 1) / kPfWarps;
    if (blocks > need) blocks = need;
    pfaffian_kernel<<<(unsigned)blocks, 32 * kPfWarps, smem, st>>>(A);
    qcs_status r = qcs_check_launch(ctx, "pfaffian_kernel");
    if (r != QCS_OK) return r;
    pair_sum_kernel<<<(unsigned)((A.W * 32 + 127) / 128), 128, 0, st>>>(A.W, A.p0, A.span, A.d_count, A.sum, L.partial,
                                                                        L.nchunks);
    return qcs_check_launch(ctx, "pair_sum_kernel");
}
