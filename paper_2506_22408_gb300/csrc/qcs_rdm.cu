// qcs_rdm.cu -- shadow estimates of Majorana correlators, the one-particle RDM
// and the particle number (Supplementary "Reduced Density Matrices", Eq.
// local_fermionic_ob_exp): for rotated Majoranas g~ = R g (R in O(2n)),
//     <g~_S> = mean_p C(2n,|S|)/C(n,|S|/2) pf( i (R G_p R^T)|_S ),   G_p = Q_p^T C_b Q_p.
// |S| = 2: pf(i X|_S) = i X_{mu nu}, so <g~_mu g~_nu> = i (2n-1) mean_p X_p,mu nu.
// |S| = 4: pf(i X|_S) = -(X_01 X_23 - X_02 X_13 + X_03 X_12), so the estimates of all
// products of four distinct Majoranas are fixed combinations of the second moments
//     S2[(mu nu), (rho sigma)] = sum_p X_p,mu nu X_p,rho sigma
// of the covariance entries: a symmetric rank-P update (K = P), the contraction that
// dominates this path.  The 1-RDM follows Eqs. (1rdm_off_diagonal) and
// (1rdm_diagonal): a~_p = (g~_2p + i g~_2p+1)/2.
//
// Kernels: rdm_cov_kernel (warp per snapshot: X_p = (Q' R^T)^T J (Q' R^T) from the
// stored rows Qt in fixed point, upper triangle to global), rdm_colsum_kernel
// (deterministic column sums), rdm_slice_kernel and rdm_tc_moment_kernel (S2 on the BF16
// tensor cores by error-free slicing; rdm_syrk_kernel, FP64, takes its place when a
// covariance is not finite), rdm_finalize_kernel (gam2, rdm1, particle number, gam4 from
// the reduced S2).  n = 16, P = 60000: 16.9 ms with the FP64 update (FP64 pipe bound) and
// 1.9 ms now, of which the moments 0.87 ms (records from L2 at 3.6 TB/s, two stages in
// flight) and the covariances 0.76 ms (integer multiplies 69 %, shared memory 65 %).
#include "qcs_fixed.cuh"
#include "qcs_internal.h"
#include "qcs_tc.cuh"

namespace {

constexpr int kTile = 32;     // S2 tile edge (small tiles: less work in the lower halves of diagonal tiles)
constexpr int kTThreads = 64; // threads per S2 tile: 8 x 8, each 4 x 4 entries
constexpr int kKStep = 16;    // snapshots staged per step
constexpr int kColRows = 256; // rows per column-sum partial (at least)
constexpr int64_t kMBatch = 65536;  // snapshots whose slices are held at once, at most (0.47 GB at n = 16)

// Upper-triangle pair index of (mu, nu), mu < nu < N2, in row-major order.
__host__ __device__ __forceinline__ int pair_rank(int mu, int nu, int N2) {
    return mu * N2 - mu * (mu + 1) / 2 + (nu - mu - 1);
}

// X_p for every snapshot (warp per snapshot), FP64 packed upper triangle to Gu, and the
// largest upper word of |X| over all of them to *d_max.
//
// Q' (and R) are held as fixed point (qcs_fixed.cuh: one scale per matrix, limbs of 29 bits):
// the products then run on the integer pipe, three IMAD.WIDE (12 clocks per 32 of them)
// where the FP64 pipe takes 76, and are exact to 2^-57 of the matrix scale; the two limbs
// of an entry are one 8-byte load.  A snapshot or rotation with a non-finite entry takes
// the FP64 loops (NaN and infinity reach the same outputs).
__global__ void rdm_cov_kernel(int n, int64_t P, const cd *__restrict__ Qt, const double *__restrict__ R,
                               double *__restrict__ Gu, unsigned *__restrict__ d_max) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned rmax_s;
    const int N2 = 2 * n, npair = N2 * (N2 - 1) / 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int mats = R ? 2 : 1;
    // the rotation as limbs (per block), then per warp Q' and, with a rotation, Q' R^T
    fxl *Rx = reinterpret_cast<fxl *>(smem_raw);
    unsigned char *mine = smem_raw + ((R ? 1 : 0) + (size_t)warp * mats) * N2 * N2 * sizeof(double);
    double *Qp = reinterpret_cast<double *>(mine), *X = Qp + N2 * N2;
    fxl *Qx = reinterpret_cast<fxl *>(mine);
    long long *Yv = reinterpret_cast<long long *>(X);
    int fR = 0;
    unsigned rmax = 0u;
    if (R) {
        if (threadIdx.x == 0) rmax_s = 0u;
        __syncthreads();
        unsigned k = 0u;
        for (int e = threadIdx.x; e < N2 * N2; e += blockDim.x) {
            const unsigned h = (unsigned)__double2hiint(R[e]) & 0x7fffffffu;
            k = h > k ? h : k;
        }
        atomicMax(&rmax_s, k);
        __syncthreads();
        rmax = rmax_s;
        fR = 57 + 1022 - (int)(rmax >> 20);
        if (rmax < 0x7ff00000u)
            for (int e = threadIdx.x; e < N2 * N2; e += blockDim.x) Rx[e] = fx_split<29>(fx_of1(R[e], fR));
        __syncthreads();
    }
    unsigned top = 0u;
    for (int64_t p = (int64_t)blockIdx.x * wpb + warp; p < P; p += (int64_t)gridDim.x * wpb) {
        const cd *q = Qt + p * N2 * n;
        double *out = Gu + p * npair;
        unsigned k = 0u;
        for (int e = lane; e < N2 * n; e += 32) k = max(k, pivot_key(q[e]));
        k = __reduce_max_sync(QCS_FULL, k);
        if (k < 0x7ff00000u && rmax < 0x7ff00000u) {
            int f = 57 + 1022 - (int)(k >> 20);  // |q| 2^f < 2^57
            for (int e = lane; e < N2 * n; e += 32) {  // Q'[c][2k] = Re Qt[c][k], Q'[c][2k+1] = -Im Qt[c][k]
                const cd v = q[e];
                Qx[2 * e] = fx_split<29>(fx_of1(v.x, f));
                Qx[2 * e + 1] = fx_split<29>(-fx_of1(v.y, f));
            }
            __syncwarp();
            if (R) {  // Q' R^T, then its largest entry to 57 bits again
                unsigned t = 0u;
                for (int e = lane; e < N2 * N2; e += 32) {
                    const int c = e / N2, mu = e - c * N2;
                    fxacc s = {0, fx_half<29>(58)};
                    for (int kk = 0; kk < N2; ++kk) fx_mac(s, Qx[c * N2 + kk], Rx[mu * N2 + kk]);
                    const long long v = fx_value<29>(s, 58);  // worth v 2^{58-f-fR}
                    Yv[e] = v;
                    t |= (unsigned)abs((int)(v >> 32));
                }
                const int b = fx_top_bits(__reduce_or_sync(QCS_FULL, t));
                f += fR - 58 + 57 - b;
                for (int e = lane; e < N2 * N2; e += 32) Qx[e] = fx_split<29>(fx_shift1(Yv[e], 57 - b));
                __syncwarp();
            }
            // X_p[mu][nu] = sum_j Y[2j][mu] Y[2j+1][nu] - Y[2j+1][mu] Y[2j][nu]   (Y^T J Y)
            int mu = 0, first = 0;  // rows of the upper triangle, the lanes' entries in order
            for (int t = lane; t < npair; t += 32) {
                while (t >= first + N2 - 1 - mu) {
                    first += N2 - 1 - mu;
                    ++mu;
                }
                const int nu = mu + 1 + t - first;
                fxacc s = {0, fx_half<29>(58)};
                const fxl *a = Qx + mu, *b = Qx + nu;
#pragma unroll 4
                for (int j = 0; j < n; ++j) {
                    fx_mac(s, a[0], b[N2]);
                    fx_mac(s, fx_neg(a[N2]), b[0]);
                    a += 2 * N2;
                    b += 2 * N2;
                }
                const double v = fx_f64(fx_value<29>(s, 58), 58 - 2 * f);
                top = max(top, (unsigned)__double2hiint(v) & 0x7fffffffu);
                out[t] = v;
            }
            __syncwarp();
            continue;
        }
        for (int e = lane; e < N2 * n; e += 32) {
            const int c = e / n, kk = e - c * n;
            const cd v = q[e];
            Qp[c * N2 + 2 * kk] = v.x;
            Qp[c * N2 + 2 * kk + 1] = -v.y;
        }
        __syncwarp();
        const double *Y = Qp;
        if (R) {
            for (int e = lane; e < N2 * N2; e += 32) {
                const int c = e / N2, mu = e - c * N2;
                double s = 0.0;
                for (int kk = 0; kk < N2; ++kk) s = fma(Qp[c * N2 + kk], R[mu * N2 + kk], s);
                X[e] = s;
            }
            __syncwarp();
            Y = X;
        }
        for (int t = lane; t < npair; t += 32) {
            int mu = 0, rem = t;
            while (rem >= N2 - 1 - mu) {
                rem -= N2 - 1 - mu;
                ++mu;
            }
            const int nu = mu + 1 + rem;
            double s = 0.0;
            for (int j = 0; j < n; ++j) {
                s = fma(Y[(2 * j) * N2 + mu], Y[(2 * j + 1) * N2 + nu], s);
                s = fma(-Y[(2 * j + 1) * N2 + mu], Y[(2 * j) * N2 + nu], s);
            }
            top = max(top, (unsigned)__double2hiint(s) & 0x7fffffffu);
            out[t] = s;
        }
        __syncwarp();
    }
    top = __reduce_max_sync(QCS_FULL, top);
    if (lane == 0 && top) atomicMax(d_max, top);
}

// part[r][t] = sum of Gu[p][t] over the rows p of block-row r (rows per block-row each).
__global__ void rdm_colsum_kernel(int64_t P, int npair, int64_t rows, const double *__restrict__ Gu,
                                  double *__restrict__ part) {
    const int64_t r = blockIdx.y;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= npair) return;
    const int64_t p0 = r * rows, p1 = p0 + rows < P ? p0 + rows : P;
    double s = 0.0;
    for (int64_t p = p0; p < p1; ++p) s += Gu[p * npair + t];
    part[r * npair + t] = s;
}

// part[0][t] = sum over the block-rows r of part[r][t], in order, four at a time (the sums in
// one thread per output took rdm_finalize_kernel 0.3 ms of dependent FP64 additions).
__global__ void rdm_colfold_kernel(int npair, int nrow, double *__restrict__ part) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= npair) return;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int r = 0; r < nrow; r += 4)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (r + k < nrow) s[k] += part[(size_t)(r + k) * npair + t];
    part[t] = (s[0] + s[1]) + (s[2] + s[3]);
}

// ---- second moments on tensor cores
//
// S2 = sum_p x_p x_p^T is a symmetric rank-P update of npair x npair FP64 entries (npair =
// 496 at n = 16).  With one scale 2^E for all entries (|x| <= 1 for orthogonal snapshots;
// the largest entry is known from rdm_cov_kernel) the entries are cut into seven balanced
// 8-bit slices (qcs_ozaki.cuh: the slices reproduce x to 2^-56 2^E), and the 28 slice
// products of the leading levels run on tcgen05: 128 snapshots of a level add up to at
// most 7 * 128 * 128^2 < 2^24, exact in FP32, after which the level sums are added to
// integers: the first five levels exactly in units of 2^{2E-46} (64 bits), the last two in
// units of 2^{2E-54} (32 bits; the last level rounded to that once per 128 snapshots).
// FP64 sums round at 2^-53 of partial sums of up to P / 31.
//
// Bounds: 28 products x 2 npair (npair + 1) / 2 P BF16 flops = 0.83 PFLOP / 1000 at n = 16,
// P = 60000: 0.44 ms at 1.9 PFLOP/s; a block's operands pass through shared memory at 86 KB
// per 32 snapshots, about 3.2 GB from L2 in all.

constexpr int kMRows = 128, kMCols = 64, kMK = 32;          // output tile, snapshots per stage
constexpr int kMSlab = kMCols * kMK * 2;                     // one slice of 64 rows x 32 snapshots: 4 KB
constexpr int kMRec = qcs_oz::kSlices * kMSlab;              // ... all slices
constexpr int kMStage = 3 * kMRec;                           // A (two row blocks) and B of a stage: 84 KB
constexpr int kMStagesPerSum = 4;                            // 128 snapshots per exact sum
constexpr uint32_t kMWait = 1u << 26;                        // bounded mbarrier waits
constexpr unsigned kNonFinite = 0x7ff00000u;

// Row scale exponent from the upper word of the largest |x| (as qcs_oz::row_exp_of).
__device__ __forceinline__ int moment_exp(unsigned hi) { return (int)((hi + (1u << 14) + 1u) >> 20) - 1022; }

// Slices of x_p, p0 <= p < p0 + 32 nkb: record (rb, kb) holds 64 pair rows x 32 snapshots as
// K-major core matrices, the seven slices in order; rows and snapshots beyond the data are
// zero.  Block: one record, thread (row, group of eight snapshots).
__global__ void __launch_bounds__(256) rdm_slice_kernel(int64_t P, int64_t p0, int npair, int nkb,
                                                        const double *__restrict__ Gu,
                                                        const unsigned *__restrict__ d_max,
                                                        unsigned char *__restrict__ rec) {
    __shared__ double xs[kMK][kMCols + 1];
    const unsigned hi = *d_max;
    if (hi >= kNonFinite) return;
    const int E = moment_exp(hi), rb = blockIdx.y, kb = blockIdx.x;
    for (int e = threadIdx.x; e < kMK * kMCols; e += 256) {
        const int k = e / kMCols, r = e - k * kMCols, t = rb * kMCols + r;
        const int64_t p = p0 + (int64_t)kb * kMK + k;
        xs[k][r] = (p < P && t < npair) ? Gu[p * npair + t] : 0.0;
    }
    __syncthreads();
    const int r = threadIdx.x & 63, g = threadIdx.x >> 6;
    uint64_t u[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) u[c] = (uint64_t)qcs_oz::fixed_of(xs[8 * g + c][r], E) + qcs_oz::kDigitBias;
    unsigned char *out = rec + ((size_t)rb * nkb + kb) * kMRec + qcs_oz::kmajor16(r, 8 * g);
#pragma unroll
    for (int i = 1; i <= qcs_oz::kSlices; ++i) {
        uint4 w;
        w.x = qcs_oz::bf16x2_of(qcs_oz::slice_f32(u[0], i), qcs_oz::slice_f32(u[1], i));
        w.y = qcs_oz::bf16x2_of(qcs_oz::slice_f32(u[2], i), qcs_oz::slice_f32(u[3], i));
        w.z = qcs_oz::bf16x2_of(qcs_oz::slice_f32(u[4], i), qcs_oz::slice_f32(u[5], i));
        w.w = qcs_oz::bf16x2_of(qcs_oz::slice_f32(u[6], i), qcs_oz::slice_f32(u[7], i));
        *reinterpret_cast<uint4 *>(out + (size_t)(i - 1) * kMSlab) = w;
    }
}

// One 128 x 64 tile of S2 over a range of 128-snapshot chunks (block (tile, split)); the
// eight warps read the accumulators, one thread copies the records (two stages in flight)
// and issues the MMAs: per A slice i the B slices j = 1 .. 8 - i as operands of up to 256
// rows, slice j into the 64 columns of level i + j.  Adds to the partials when add is set.
__global__ void __launch_bounds__(256, 1) rdm_tc_moment_kernel(int npair, int nkb, int nchunk, int cps,
                                                               const unsigned char *__restrict__ rec,
                                                               const unsigned *__restrict__ d_max, int add,
                                                               double *__restrict__ S2p, unsigned *status) {
    using namespace qcs_tc;
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ uint32_t tmem_base;
    __shared__ __align__(8) uint64_t full[2], done[2], summed;
    __shared__ int bad;
    const unsigned hi = *d_max;
    if (hi >= kNonFinite) return;  // block-uniform, nothing allocated yet
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // tiles (ti, tj) that reach the upper triangle: tj >= 2 ti
    const int ncol = (npair + kMCols - 1) / kMCols;
    int lin = blockIdx.x, ti = 0;
    while (lin >= ncol - 2 * ti) {
        lin -= ncol - 2 * ti;
        ++ti;
    }
    const int tj = 2 * ti + lin;
    const int nrb = ncol;
    const int c0 = blockIdx.y * cps, c1 = c0 + cps < nchunk ? c0 + cps : nchunk;
    const int nst = c1 > c0 ? kMStagesPerSum * (c1 - c0) : 0;
    if (!QCS_IN_BOUNDS(2 * kMStage <= (int)dyn_smem_bytes() && tj < nrb && c1 * kMStagesPerSum <= nkb, status)) return;
    if (warp == 0) {
        tmem_alloc(&tmem_base, 512);
        tmem_relinquish();
    }
    if (t == 0) {
        for (int k = 0; k < 2; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&done[k], 1);
        }
        mbar_init(&summed, 1);
        bad = 0;
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tm = tmem_base;
    const bool two = 2 * ti + 1 < nrb;  // the tile's second row block exists (else rows are not used)
    bool ok = true;
    int loads = 0;  // stages whose copies thread 0 has issued
    // thread 0: the records of stage st into its slot, once the MMAs that read the slot are done
    auto load = [&](int st) {
        const int s = st & 1;
        if (st >= 2 && !mbar_wait_bounded(&done[s], (uint32_t)((st - 2) >> 1) & 1u, kMWait)) return false;
        unsigned char *A = sm + (size_t)s * kMStage, *B = A + 2 * kMRec;
        const int kb = c0 * kMStagesPerSum + st;
        const unsigned char *a0 = rec + ((size_t)(2 * ti) * nkb + kb) * kMRec;
        const unsigned char *a1 = rec + ((size_t)(two ? 2 * ti + 1 : 2 * ti) * nkb + kb) * kMRec;
        mbar_expect_tx(&full[s], kMStage);
        for (int i = 0; i < qcs_oz::kSlices; ++i) {  // slice i: rows 0-63, then 64-127
            bulk_copy(A + (size_t)i * 2 * kMSlab, a0 + (size_t)i * kMSlab, kMSlab, &full[s]);
            bulk_copy(A + (size_t)i * 2 * kMSlab + kMSlab, a1 + (size_t)i * kMSlab, kMSlab, &full[s]);
        }
        bulk_copy(B, rec + ((size_t)tj * nkb + kb) * kMRec, kMRec, &full[s]);
        loads = st + 1;
        return true;
    };
    long long acc[32];  // in units of 2^{2E-46}
    int low[32];        // ... of 2^{2E-54}
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        acc[c] = 0;
        low[c] = 0;
    }
    volatile int *badv = &bad;
    if (t == 0 && nst > 0 && !(load(0) && (nst < 2 || load(1)))) *badv = 1;
    for (int st = 0; st < nst; ++st) {
        const int s = st & 1;
        if (t == 0 && !*badv) {
            bool go = mbar_wait_bounded(&full[s], (uint32_t)(st >> 1) & 1u, kMWait);
            if (go) {
                fence_after_sync();
                const unsigned char *A = sm + (size_t)s * kMStage, *B = A + 2 * kMRec;
                const bool first = (st % kMStagesPerSum) == 0;
                for (int i = 1; i <= qcs_oz::kSlices; ++i)
                    for (int ks = 0; ks < 2; ++ks) {
                        const uint64_t ad = desc_kmajor(A + (size_t)(i - 1) * 2 * kMSlab + 256 * ks, 128, 512);
                        for (int j = 1; j <= 8 - i; j += 4) {
                            const int nj = 8 - i - j + 1 < 4 ? 8 - i - j + 1 : 4;
                            const uint64_t bd = desc_kmajor(B + (size_t)(j - 1) * kMSlab + 256 * ks, 128, 512);
                            mma_f16(tm + (uint32_t)(kMCols * (i + j - 2)), ad, bd, idesc_bf16(kMRows, kMCols * nj),
                                    first && i == 1 && ks == 0 ? 0u : 1u);
                        }
                    }
                mma_commit(&done[s]);
                if ((st + 1) % kMStagesPerSum == 0) mma_commit(&summed);
                // the other slot's next records, once its MMAs (the stage before) are done
                if (st >= 1 && st + 1 < nst) go = load(st + 1);
            }
            if (!go) *badv = 1;
        }
        if ((st + 1) % kMStagesPerSum == 0) {
            // the sums of 128 snapshots: this thread's lane (row) and 32 columns of every level
            const uint32_t ph = (uint32_t)(st / kMStagesPerSum) & 1u;
            bool w = false;
            for (int tries = 0; tries < 64 && !w && !*badv; ++tries) w = mbar_wait_bounded(&summed, ph, kMWait >> 6);
            ok = __syncthreads_and(w);
            if (!ok) break;
            __syncwarp();
            fence_after_sync();
            const uint32_t ta = tm + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(32 * (warp >> 2));
#pragma unroll
            for (int cb = 0; cb < 8; ++cb) {
                float v[qcs_oz::kLevels][4];
#pragma unroll
                for (int L = 0; L < qcs_oz::kLevels; ++L) tmem_ld4(ta + (uint32_t)(kMCols * L + 4 * cb), v[L]);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    int x[qcs_oz::kLevels];
#pragma unroll
                    for (int L = 0; L < qcs_oz::kLevels; ++L) x[L] = __float2int_rn(v[L][c]);
                    long long z = acc[4 * cb + c] + (long long)x[4];
                    low[4 * cb + c] += x[5] + ((x[6] + 128) >> 8);
                    z = mad_wide(x[3], 256, z);
                    z = mad_wide(x[2], 65536, z);
                    z = mad_wide(x[1], 16777216, z);
                    acc[4 * cb + c] = z + ((long long)x[0] << 32);
                }
            }
            if (((st / kMStagesPerSum) & 63) == 63) {  // before the low words can overflow
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    acc[c] += low[c] >> 8;
                    low[c] &= 255;
                }
            }
            fence_before_sync();
            __syncthreads();  // the next chunk's first MMAs overwrite the accumulators
            fence_after_sync();
        }
    }
    if (!ok && t == 0) {
        raise_status(status, QCS_ERR_TIMEOUT);
        // let copies and MMAs in flight land before the shared and tensor memory go
        for (int st = loads > 2 ? loads - 2 : 0; st < loads; ++st) {
            mbar_wait_bounded(&full[st & 1], (uint32_t)(st >> 1) & 1u, kMWait);
            mbar_wait_bounded(&done[st & 1], (uint32_t)(st >> 1) & 1u, 1u << 20);
        }
    }
    const int E2 = 2 * moment_exp(hi) - 46;
    const int i = ti * kMRows + 32 * (warp & 3) + lane;
    double *out = S2p + (size_t)blockIdx.y * npair * npair + (size_t)i * npair;
    if (ok && i < npair)
#pragma unroll
        for (int c = 0; c < 32; ++c) {
            const int j = tj * kMCols + 32 * (warp >> 2) + c;
            if (j < npair && i <= j) {
                const double v = fx_f64(acc[c], E2) + fx_f64(low[c], E2 - 8);
                out[j] = add ? out[j] + v : v;
            }
        }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == 0) tmem_dealloc(tm, 512);
}

// S2 partials: block (ti, tj, ks) with ti <= tj computes the 32 x 32 tile
// sum_{p in range ks} Gu[p][i] Gu[p][j]; each of the 64 threads owns 4 x 4 entries.
// Snapshots with a non-finite covariance only (NaN and infinity have no slices); otherwise it
// returns at once.
__global__ void __launch_bounds__(kTThreads) rdm_syrk_kernel(int64_t P, int npair, int ntile, int64_t krange,
                                                             const double *__restrict__ Gu,
                                                             const unsigned *__restrict__ d_max,
                                                             double *__restrict__ S2p) {
    if (*d_max < kNonFinite) return;
    __shared__ double As[kKStep][kTile + 1];
    __shared__ double Bs[kKStep][kTile + 1];
    // upper-triangle tile (ti, tj) from the linear block index
    int lin = blockIdx.x, ti = 0;
    while (lin >= ntile - ti) {
        lin -= ntile - ti;
        ++ti;
    }
    const int tj = ti + lin;
    const int64_t ks = blockIdx.y;
    const int64_t p0 = ks * krange, p1 = p0 + krange < P ? p0 + krange : P;
    const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
    const int i0 = ti * kTile, j0 = tj * kTile;
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = 0.0;
    for (int64_t pb = p0; pb < p1; pb += kKStep) {
        for (int e = threadIdx.x; e < kKStep * kTile; e += blockDim.x) {
            const int kk = e / kTile, col = e - kk * kTile;
            const int64_t p = pb + kk;
            const bool in = p < p1;
            As[kk][col] = (in && i0 + col < npair) ? Gu[p * npair + i0 + col] : 0.0;
            Bs[kk][col] = (in && j0 + col < npair) ? Gu[p * npair + j0 + col] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kKStep; ++kk) {
            double a[4], bb[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] = As[kk][ty + 8 * u];
                bb[u] = Bs[kk][tx + 8 * u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v] = fma(a[u], bb[v], acc[u][v]);
        }
        __syncthreads();
    }
    double *out = S2p + (size_t)ks * npair * npair;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int i = i0 + ty + 8 * u, j = j0 + tx + 8 * v;
            if (i < npair && j < npair && i <= j) out[(size_t)i * npair + j] = acc[u][v];
        }
}

inline double binom_d(int n, int k) {
    if (k < 0 || k > n) return 0.0;
    double r = 1.0;
    for (int i = 1; i <= k; ++i) r = r * (double)(n - k + i) / (double)i;
    return r;
}

// Lexicographic rank of the 4-subset a < b < c < d of {0..N-1}.
__device__ __forceinline__ int rank4(int a, int b, int c, int d, int N) {
    auto c4 = [](int x) { return (unsigned)(x * (x - 1) * (x - 2) * (x - 3)) / 24u; };  // x <= 48
    const int x = N - 1 - b, y = N - 1 - c;
    return (int)(c4(N) - 1u - c4(N - 1 - a) - (unsigned)(x * (x - 1) * (x - 2)) / 6u - (unsigned)(y * (y - 1)) / 2u -
                 (unsigned)(N - 1 - d));
}

// S2 entry (pair i, pair j) summed over the snapshot ranges (only i <= j is stored).
__device__ __forceinline__ double s2_at(const double *S2p, int nks, int npair, int i, int j) {
    if (i > j) {
        int t = i;
        i = j;
        j = t;
    }
    double s = 0.0;
    for (int k = 0; k < nks; ++k) s += S2p[(size_t)k * npair * npair + (size_t)i * npair + j];
    return s;
}

__global__ void rdm_finalize_kernel(int n, int64_t P, const double *__restrict__ part,
                                    const double *__restrict__ S2p, int nks, double K2, double K4,
                                    double *__restrict__ gam2, double *__restrict__ gam4, cd *__restrict__ rdm1,
                                    double *__restrict__ npart) {
    const int N2 = 2 * n, npair = N2 * (N2 - 1) / 2;
    const double invP = 1.0 / (double)P;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x;
    auto mean_pair = [&](int mu, int nu) {  // K2 mean_p X[mu][nu], antisymmetric, 0 on the diagonal
        if (mu == nu) return 0.0;
        const int lo = mu < nu ? mu : nu, hi = mu < nu ? nu : mu;
        const int t = pair_rank(lo, hi, N2);
        const double s = part[t] * (K2 * invP);
        return mu < nu ? s : -s;
    };
    if (gam2)
        for (int e = tid; e < N2 * N2; e += nthr) gam2[e] = mean_pair(e / N2, e % N2);
    if (rdm1 || npart) {
        // <g_mu g_nu> = i gam2[mu][nu];  a_p^dag a_q = (1/4)(g_2p - i g_2p+1)(g_2q + i g_2q+1)
        for (int e = tid; e < n * n; e += nthr) {
            const int p = e / n, q = e - p * n;
            cd d;
            if (p == q) {
                d = cmk(0.5 * (1.0 - mean_pair(2 * p, 2 * p + 1)), 0.0);
            } else {
                const double g00 = mean_pair(2 * p, 2 * q), g01 = mean_pair(2 * p, 2 * q + 1);
                const double g10 = mean_pair(2 * p + 1, 2 * q), g11 = mean_pair(2 * p + 1, 2 * q + 1);
                // (1/4)(i g00 + i (i g01) - i (i g10) + i g11) = (1/4)(-g01 + g10, g00 + g11)
                d = cmk(0.25 * (g10 - g01), 0.25 * (g00 + g11));
            }
            if (rdm1) rdm1[e] = d;
        }
        if (npart && tid == 0) {
            double s = 0.0;
            for (int p = 0; p < n; ++p) s += 0.5 * (1.0 - mean_pair(2 * p, 2 * p + 1));
            *npart = s;
        }
    }
    if (gam4 && S2p) {
        // one thread per ordered pair of index pairs (mu<nu), (rho<sigma) with nu < rho
        for (long long e = tid; e < (long long)npair * npair; e += nthr) {
            const int t1 = (int)(e / npair), t2 = (int)(e - (long long)t1 * npair);
            int mu = 0, rem = t1;
            while (rem >= N2 - 1 - mu) {
                rem -= N2 - 1 - mu;
                ++mu;
            }
            const int nu = mu + 1 + rem;
            int rho = 0;
            rem = t2;
            while (rem >= N2 - 1 - rho) {
                rem -= N2 - 1 - rho;
                ++rho;
            }
            const int sg = rho + 1 + rem;
            if (nu >= rho) continue;
            const double v = s2_at(S2p, nks, npair, t1, t2) -
                             s2_at(S2p, nks, npair, pair_rank(mu, rho, N2), pair_rank(nu, sg, N2)) +
                             s2_at(S2p, nks, npair, pair_rank(mu, sg, N2), pair_rank(nu, rho, N2));
            gam4[rank4(mu, nu, rho, sg, N2)] = -K4 * v * invP;
        }
    }
}

}  // namespace

extern "C" qcs_status qcs_shadow_rdm(qcs_ctx *ctx, const qcs_snapshots *s, const double *d_R, double *d_gam2,
                                     double *d_gam4, double *d_rdm1, double *d_npart, void *stream) {
    QcsRange range_("qcs_shadow_rdm");
    if (!ctx) return QCS_ERR_ARG;
    if (!s) return qcs_fail(ctx, QCS_ERR_ARG, "null snapshot set");
    if (s->device != ctx->device) return qcs_fail(ctx, QCS_ERR_ARG, "snapshot set lives on another device");
    if (s->P < 1) return qcs_fail(ctx, QCS_ERR_ARG, "the snapshot set is empty");
    const int n = s->n, N2 = 2 * n, npair = N2 * (N2 - 1) / 2;
    if (d_gam4 && n < 2) return qcs_fail(ctx, QCS_ERR_ARG, "four-Majorana estimates need n >= 2");
    cudaStream_t st = (cudaStream_t)stream;
    DeviceGuard g(ctx->device);
    const int64_t P = s->P;
    int64_t rows = kColRows;
    if ((P + rows - 1) / rows > 4096) rows = (P + 4095) / 4096;  // at most 4096 block-rows (grid.y)
    const int nrow = (int)((P + rows - 1) / rows);
    // split the snapshot range of the S2 update so that the grid covers the GPU (one block
    // per SM); the slices of at most kMBatch snapshots at a time
    const int ntile = (npair + kTile - 1) / kTile;
    const int nut = ntile * (ntile + 1) / 2;
    const int ncol = (npair + kMCols - 1) / kMCols;
    int ntc = 0;
    for (int ti = 0; 2 * ti < ncol; ++ti) ntc += ncol - 2 * ti;
    constexpr int64_t kSum = (int64_t)kMStagesPerSum * kMK;
    const size_t b_gu = align16(sizeof(double) * (size_t)P * npair);
    const size_t b_part = align16(sizeof(double) * (size_t)nrow * npair);
    int nks = 1;
    int64_t batch = 0;
    size_t b_s2 = 0;
    auto layout = [&](int64_t sums) {
        batch = sums * kSum;
        if (d_gam4) {
            nks = ctx->num_sms / ntc;
            if (nks > sums) nks = (int)sums;
            if (nks < 1) nks = 1;
        }
        b_s2 = d_gam4 ? align16(sizeof(double) * (size_t)nks * npair * npair) : 0;
        return 16 + b_gu + b_part + b_s2 + (d_gam4 ? (size_t)ncol * (size_t)(batch / kMK) * kMRec : 0);
    };
    void *base = nullptr;
    const int64_t most = P < kMBatch ? (P + kSum - 1) / kSum : kMBatch / kSum;
    qcs_status ws = qcs_workspace_batched(ctx, most, d_gam4 ? 1 : most, layout, &base, st);
    if (ws != QCS_OK) return ws;
    const int64_t krange = ((P + nks - 1) / nks + kKStep - 1) / kKStep * kKStep;
    unsigned *d_max = (unsigned *)base;
    double *Gu = (double *)((char *)base + 16);
    double *part = (double *)((char *)base + 16 + b_gu);
    double *S2p = d_gam4 ? (double *)((char *)base + 16 + b_gu + b_part) : nullptr;
    unsigned char *rec = (unsigned char *)base + 16 + b_gu + b_part + b_s2;
    if (cudaMemsetAsync(d_max, 0, sizeof(unsigned), st) != cudaSuccess) return qcs_fail(ctx, QCS_ERR_CUDA, "rdm reset");
    {
        const int wpb = 4;
        const size_t smem = ((d_R ? 1 : 0) + (size_t)wpb * (d_R ? 2 : 1)) * N2 * N2 * sizeof(double);
        if (qcs_set_smem(ctx, (const void *)rdm_cov_kernel, smem) != QCS_OK) return QCS_ERR_CUDA;
        int64_t blocks = (P + wpb - 1) / wpb;
        if (blocks > (int64_t)ctx->num_sms * 16) blocks = (int64_t)ctx->num_sms * 16;
        rdm_cov_kernel<<<(unsigned)blocks, wpb * 32, smem, st>>>(n, P, s->Qt, d_R, Gu, d_max);
        qcs_status r = qcs_check_launch(ctx, "rdm_cov_kernel");
        if (r != QCS_OK) return r;
    }
    rdm_colsum_kernel<<<dim3((unsigned)((npair + 127) / 128), (unsigned)nrow), 128, 0, st>>>(P, npair, rows, Gu,
                                                                                            part);
    qcs_status r = qcs_check_launch(ctx, "rdm_colsum_kernel");
    if (r != QCS_OK) return r;
    rdm_colfold_kernel<<<(unsigned)((npair + 63) / 64), 64, 0, st>>>(npair, nrow, part);
    r = qcs_check_launch(ctx, "rdm_colfold_kernel");
    if (r != QCS_OK) return r;
    if (d_gam4) {
        if (cudaMemsetAsync(S2p, 0, b_s2, st) != cudaSuccess) return qcs_fail(ctx, QCS_ERR_CUDA, "S2 reset");
        if (qcs_set_smem(ctx, (const void *)rdm_tc_moment_kernel, 2 * kMStage) != QCS_OK) return QCS_ERR_CUDA;
        qcs_prof_begin(ctx, st);
        for (int64_t p0 = 0; p0 < P; p0 += batch) {
            const int64_t here = P - p0 < batch ? P - p0 : batch;
            const int nchunk = (int)((here + kSum - 1) / kSum), nkb = nchunk * kMStagesPerSum;
            const int cps = (nchunk + nks - 1) / nks;
            rdm_slice_kernel<<<dim3((unsigned)nkb, (unsigned)ncol), 256, 0, st>>>(P, p0, npair, nkb, Gu, d_max, rec);
            r = qcs_check_launch(ctx, "rdm_slice_kernel");
            if (r != QCS_OK) return r;
            rdm_tc_moment_kernel<<<dim3((unsigned)ntc, (unsigned)nks), 256, 2 * kMStage, st>>>(
                npair, nkb, nchunk, cps, rec, d_max, p0 > 0 ? 1 : 0, S2p, ctx->d_status);
            r = qcs_check_launch(ctx, "rdm_tc_moment_kernel");
            if (r != QCS_OK) return r;
        }
        qcs_prof_end(ctx, st);
        rdm_syrk_kernel<<<dim3((unsigned)nut, (unsigned)nks), kTThreads, 0, st>>>(P, npair, ntile, krange, Gu, d_max,
                                                                                 S2p);
        r = qcs_check_launch(ctx, "rdm_syrk_kernel");
        if (r != QCS_OK) return r;
    }
    // channel weights
    const double K2 = binom_d(N2, 2) / binom_d(n, 1), K4 = n >= 2 ? binom_d(N2, 4) / binom_d(n, 2) : 0.0;
    int64_t fin = d_gam4 ? ((int64_t)npair * npair + 255) / 256 : 4;
    if (fin > (int64_t)ctx->num_sms * 8) fin = (int64_t)ctx->num_sms * 8;
    rdm_finalize_kernel<<<(unsigned)fin, 256, 0, st>>>(n, P, part, S2p, nks, K2, K4, d_gam2, d_gam4,
                                                       (cd *)d_rdm1, d_npart);
    return qcs_check_launch(ctx, "rdm_finalize_kernel");
}

extern "C" double qcs_shadow_rdm_flops(int n, int64_t P) {
    if (n < 2 || n > QCS_MAX_N || P < 1) return 0.0;
    const double npair = (double)(2 * n) * (2 * n - 1) / 2.0;
    // the symmetric rank-P update of the pair moments (upper triangle incl. diagonal)
    return 2.0 * (double)P * npair * (npair + 1.0) / 2.0;
}
