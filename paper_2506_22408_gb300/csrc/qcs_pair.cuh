// qcs_pair.cuh -- per-pair device building blocks shared by the overlap and
// adjoint kernels: the packed-pair table, the congruence T = Ut Qt^T and the
// selected covariance B^(s) of Eqs. (a_mat), (b_mat).
#pragma once
#include "qcs_common.cuh"

constexpr int kMaxNB = 8;  // node matrices per warp round, at most

// tab[t] = (b << 8) | a for t = b(b-1)/2 + a, a < b  (pairs in packed-upper order).
__device__ inline void build_pair_table(uint16_t *tab, int count) {
    for (int t = threadIdx.x; t < count; t += blockDim.x) {
        int b = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)t)) * 0.5f);
        while (b * (b - 1) / 2 > t) --b;
        while ((b + 1) * b / 2 <= t) ++b;
        int a = t - b * (b - 1) / 2;
        tab[t] = (uint16_t)((b << 8) | a);
    }
}

// Shared-memory row strides: one complex entry of padding per row keeps rows
// that different lanes read in the same step on different banks.
__host__ __device__ __forceinline__ int ld_ut(int n) { return n + 1; }   // Ut: n rows of n
__host__ __device__ __forceinline__ int ld_qt(int n) { return n + 1; }   // Qt: 2n rows of n
__host__ __device__ __forceinline__ int ld_t(int n) { return 2 * n + 1; }  // T: n rows of 2n

// T[j][c] = sum_k Ut[j][k] Qt[c][k]  (n x 2n; entries spread over the nthr
// threads that share the pair, lane = this thread's index among them)
__device__ inline void build_T(int n, const cd *__restrict__ Uts, const cd *__restrict__ Qs, cd *__restrict__ Ts,
                               int lane, int nthr = 32) {
    const int n2 = 2 * n, lu = ld_ut(n), lq = ld_qt(n), lt = ld_t(n);
    for (int e = lane; e < n * n2; e += nthr) {
        int j = e / n2, c = e - j * n2;
        const cd *ur = Uts + j * lu, *qr = Qs + c * lq;
        cd s = cmk(0.0, 0.0);
        for (int k = 0; k < n; ++k) cfma(s, ur[k], qr[k]);
        Ts[j * lt + c] = s;
    }
}

// T from walker rows in echelon form (see qcs_walker.cu): row j < ne of Ut is zero in
// columns k < j, row ne + j' zero in columns [ne, ne + j'); those products are skipped.
// With 2n = 32 every warp pass covers one row, so the loop bounds are warp-uniform.
__device__ inline void build_T_echelon(int n, int ne, const cd *__restrict__ Uts, const cd *__restrict__ Qs,
                                       cd *__restrict__ Ts, int lane, int nthr = 32) {
    const int n2 = 2 * n, lu = ld_ut(n), lq = ld_qt(n), lt = ld_t(n);
    for (int e = lane; e < n * n2; e += nthr) {
        const int j = e / n2, c = e - j * n2;
        const cd *ur = Uts + j * lu, *qr = Qs + c * lq;
        cd s = cmk(0.0, 0.0);
        if (j < ne) {
            for (int k = j; k < n; ++k) cfma(s, ur[k], qr[k]);
        } else {
            for (int k = 0; k < ne; ++k) cfma(s, ur[k], qr[k]);
            for (int k = j; k < n; ++k) cfma(s, ur[k], qr[k]);  // j = ne + j'
        }
        Ts[j * lt + c] = s;
    }
}

// T from echelon-form walker rows for n = N (2N = 32 lanes): lane c holds row c of the
// snapshot's Qt in registers and owns column c of T.  Each complex multiply-add takes
// three real products (Gauss's 3-multiplication form): with s = re + im of both
// factors, Re = sum ur qr - sum ui qi and Im = sum us qs - sum ur qr - sum ui qi, so
// the sums us of the walker rows (Uss, per block) and qs of the snapshot row (here)
// are formed once.  The skipped zeros follow build_T_echelon, or for a walker in
// reduced form (occupied rows [I; X]: row j < ne has its one entry at column j
// among the columns k < ne) that single entry and the columns k >= ne; the row loop
// is warp-uniform and enters the unrolled k sequences by a switch, so the register
// arrays are indexed by constants.
#define QCS_T3M(K)                            \
    case K: {                                 \
        const cd u_ = ur[K];                  \
        p1 = fma(u_.x, qr[K], p1);            \
        p2 = fma(u_.y, qi[K], p2);            \
        p3 = fma(us[K], qs[K], p3);           \
    }
#define QCS_T3M1(K)                           \
    case K: {                                 \
        const cd u_ = ur[K];                  \
        p1 = fma(u_.x, qr[K], p1);            \
        p2 = fma(u_.y, qi[K], p2);            \
        p3 = fma(us[K], qs[K], p3);           \
        break;                                \
    }
// Qg holds the snapshot's rows with stride ldq (global memory or staged); rows
// j0, j0 + jstep, ... of T are formed, so that several warps can share one T.
template <int N>
__device__ inline void build_T_reg(int ne, const cd *__restrict__ Uts, const double *__restrict__ Uss,
                                   const cd *__restrict__ Qg, cd *__restrict__ Ts, int lane, bool reduced,
                                   int ldq = N, int j0 = 0, int jstep = 1) {
    static_assert(N == 16, "one lane per column of T: 2N must be the warp width");
    const int lu = ld_ut(N), lt = ld_t(N);
    double qr[N], qi[N], qs[N];
    const cd *qrow = Qg + lane * ldq;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const cd q = qrow[k];
        qr[k] = q.x;
        qi[k] = q.y;
        qs[k] = q.x + q.y;
    }
    for (int j = j0; j < N; j += jstep) {
        const cd *ur = Uts + j * lu;
        const double *us = Uss + j * lu;
        double p1 = 0.0, p2 = 0.0, p3 = 0.0;
        int kstart = j;
        if (j < ne && reduced) {
            switch (j) {  // the single entry among the columns k < ne
                QCS_T3M1(0) QCS_T3M1(1) QCS_T3M1(2) QCS_T3M1(3) QCS_T3M1(4) QCS_T3M1(5) QCS_T3M1(6) QCS_T3M1(7)
                QCS_T3M1(8) QCS_T3M1(9) QCS_T3M1(10) QCS_T3M1(11) QCS_T3M1(12) QCS_T3M1(13) QCS_T3M1(14)
                QCS_T3M1(15)
                default: break;
            }
            kstart = ne;
        }
        if (j >= ne) {
            switch (ne - 1) {  // k = ne-1 down to 0
                QCS_T3M(15) QCS_T3M(14) QCS_T3M(13) QCS_T3M(12) QCS_T3M(11) QCS_T3M(10) QCS_T3M(9) QCS_T3M(8)
                QCS_T3M(7) QCS_T3M(6) QCS_T3M(5) QCS_T3M(4) QCS_T3M(3) QCS_T3M(2) QCS_T3M(1) QCS_T3M(0)
                default: break;
            }
        }
        switch (kstart) {  // k = kstart up to N-1
            QCS_T3M(0) QCS_T3M(1) QCS_T3M(2) QCS_T3M(3) QCS_T3M(4) QCS_T3M(5) QCS_T3M(6) QCS_T3M(7)
            QCS_T3M(8) QCS_T3M(9) QCS_T3M(10) QCS_T3M(11) QCS_T3M(12) QCS_T3M(13) QCS_T3M(14) QCS_T3M(15)
            default: break;
        }
        Ts[j * lt + lane] = cmk(p1 - p2, p3 - p1 - p2);
    }
}
#undef QCS_T3M
#undef QCS_T3M1

// x * ph for a phase code ph = 0..3 (1, i, -1, -i): a swap of the parts and sign
// flips of the bit patterns, no floating-point arithmetic.
__device__ __forceinline__ cd mul_phase(cd x, unsigned ph) {
    cd r = (ph & 1u) ? cmk(x.y, x.x) : x;
    const bool fre = ph == 1u || ph == 2u, fim = ph >= 2u;
    if (fre) r.x = __longlong_as_double(__double_as_longlong(r.x) ^ (long long)0x8000000000000000ull);
    if (fim) r.y = __longlong_as_double(__double_as_longlong(r.y) ^ (long long)0x8000000000000000ull);
    return r;
}

// Stage a snapshot's rows Qt (2n x n, global) into padded shared rows.
__device__ inline void load_Qt(int n, const cd *__restrict__ Qg, cd *__restrict__ Qs, int lane, int nthr = 32) {
    const int lq = ld_qt(n);
    for (int e = lane; e < 2 * n * n; e += nthr) {
        int c = e / n, k = e - c * n;
        Qs[c * lq + k] = Qg[e];
    }
}

__device__ __forceinline__ void pair_of(const uint16_t *tab, int t, int &a, int &b) {
    unsigned v = tab[t];
    a = v & 0xff;
    b = v >> 8;
}

// B^(s) (packed upper, m x m) from T (n x 2n).
__device__ inline void build_B(int n, int ne, const cd *__restrict__ Ts, cd *__restrict__ Bs,
                               const uint16_t *__restrict__ tab, int lane, int nthr = 32) {
    const int d = n - ne, n2 = ld_t(n);
    // occupied x occupied: complex x complex
    const int c1 = tri_count(ne);
    for (int e = lane; e < c1; e += nthr) {
        int a, b;
        pair_of(tab, e, a, b);
        const cd *Ta = Ts + a * n2, *Tb = Ts + b * n2;
        cd acc = cmk(0.0, 0.0);
        for (int k = 0; k < n; ++k) {
            cfma(acc, Ta[2 * k], Tb[2 * k + 1]);
            cfms(acc, Ta[2 * k + 1], Tb[2 * k]);
        }
        Bs[tri_index(a, b)] = acc;
    }
    // occupied x empty: complex x real.  Empty row r of mode j = ne + r/2 is
    // Re T_j (r even) or -Im T_j (r odd); the sign is applied once at the end.
    const int twod = 2 * d;
    const int c2 = ne * twod;
    for (int e = lane; e < c2; e += nthr) {
        int a = e / twod, r = e - a * twod;
        int j = ne + (r >> 1);
        bool odd = r & 1;
        const cd *Ta = Ts + a * n2, *Tj = Ts + j * n2;
        cd acc = cmk(0.0, 0.0);
        for (int k = 0; k < n; ++k) {
            cd t0 = Tj[2 * k], t1 = Tj[2 * k + 1];
            double x0 = odd ? t0.y : t0.x, x1 = odd ? t1.y : t1.x;
            crfma(acc, Ta[2 * k], x1);
            crfma(acc, Ta[2 * k + 1], -x0);
        }
        Bs[tri_index(a, ne + r)] = flip_if(acc, odd);
    }
    // empty x empty: real x real
    const int c3 = tri_count(twod);
    for (int e = lane; e < c3; e += nthr) {
        int a, b;
        pair_of(tab, e, a, b);
        const cd *Ta = Ts + (ne + (a >> 1)) * n2, *Tb = Ts + (ne + (b >> 1)) * n2;
        bool oa = a & 1, ob = b & 1;
        double acc = 0.0;
        for (int k = 0; k < n; ++k) {
            cd a0 = Ta[2 * k], a1 = Ta[2 * k + 1], b0 = Tb[2 * k], b1 = Tb[2 * k + 1];
            double xa0 = oa ? a0.y : a0.x, xa1 = oa ? a1.y : a1.x;
            double xb0 = ob ? b0.y : b0.x, xb1 = ob ? b1.y : b1.x;
            acc = fma(xa0, xb1, acc);
            acc = fma(-xa1, xb0, acc);
        }
        Bs[tri_index(ne + a, ne + b)] = cmk((oa != ob) ? -acc : acc, 0.0);
    }
}

