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

// Columns c0 .. c0+n-1 of T from n staged rows of Qt (Qs, stride ld_qt) and their
// re + im sums (qs, n x n), with three real products per complex multiply-add as in
// build_T_reg (Uss: re + im of the walker rows): Re = sum ur qr - sum ui qi,
// Im = sum us qs - sum ur qr - sum ui qi.  Walker rows in echelon form skip their zeros
// (occupied row j: columns k < j; completion row ne + j': columns ne .. ne + j' - 1);
// in reduced form (red: occupied rows [I; X] / sqrt2) an occupied row j has one entry,
// at column j, among the columns k < ne.
__device__ inline void build_T_half3(int n, int ne, bool red, const cd *__restrict__ Uts,
                                     const double *__restrict__ Uss, const cd *__restrict__ Qs,
                                     const double *__restrict__ qs, cd *__restrict__ Ts, int c0, int lane,
                                     int nthr) {
    const int lu = ld_ut(n), lq = ld_qt(n), lt = ld_t(n);
    for (int e = lane; e < n * n; e += nthr) {
        const int j = e / n, c = e - j * n;
        const cd *ur = Uts + j * lu, *qr = Qs + c * lq;
        const double *us = Uss + j * lu, *qsr = qs + c * n;
        double p1 = 0.0, p2 = 0.0, p3 = 0.0;
        int k0 = 0, k1 = 0;  // columns [k0, k1) before the tail, then [kt, n)
        int kt = j;
        if (j < ne) {
            if (red) {
                k0 = j;
                k1 = j + 1;
                kt = ne;
            }
        } else {
            k1 = ne;  // the occupied columns, then the completion's tail from j = ne + j'
        }
        for (int k = k0; k < k1; ++k) {
            const cd u = ur[k], q = qr[k];
            p1 = fma(u.x, q.x, p1);
            p2 = fma(u.y, q.y, p2);
            p3 = fma(us[k], qsr[k], p3);
        }
        for (int k = kt; k < n; ++k) {
            const cd u = ur[k], q = qr[k];
            p1 = fma(u.x, q.x, p1);
            p2 = fma(u.y, q.y, p2);
            p3 = fma(us[k], qsr[k], p3);
        }
        Ts[j * lt + c0 + c] = cmk(p1 - p2, p3 - p1 - p2);
    }
}

// x * ph for a phase code ph = 0..3 (1, i, -1, -i): a swap of the parts and sign
// flips of the bit patterns, no floating-point arithmetic.
__device__ __forceinline__ cd mul_phase(cd x, unsigned ph) {
    cd r = (ph & 1u) ? cmk(x.y, x.x) : x;
    const bool fre = ph == 1u || ph == 2u, fim = ph >= 2u;
    if (fre) r.x = __longlong_as_double(__double_as_longlong(r.x) ^ (long long)0x8000000000000000ull);
    if (fim) r.y = __longlong_as_double(__double_as_longlong(r.y) ^ (long long)0x8000000000000000ull);
    return r;
}

// Signed-permutation snapshot: row c of Qt has one nonzero entry, the phase
// code & 3 at column code >> 2, so T[j][c] = Ut[j][k_c] ph_c is a gather.
__device__ inline void build_T_gather(int n, const cd *__restrict__ Uts, const uint8_t *__restrict__ code,
                                      cd *__restrict__ Ts, int lane, int nthr = 32) {
    const int n2 = 2 * n, lu = ld_ut(n), lt = ld_t(n);
    for (int e = lane; e < n * n2; e += nthr) {
        const int j = e / n2, c = e - j * n2;
        const unsigned q = code[c];
        Ts[j * lt + c] = mul_phase(Uts[j * lu + (int)(q >> 2)], q & 3u);
    }
}

// Stage a snapshot's rows Qt (2n x n, global) into padded shared rows.
__device__ inline void load_Qt(int n, const cd *__restrict__ Qg, cd *__restrict__ Qs, int lane, int nthr = 32) {
    const int lq = ld_qt(n);
    for (int e = lane; e < 2 * n * n; e += nthr) {
        int c = e / n, k = e - c * n;
        Qs[c * lq + k] = Qg[e];
    }
}

// Stage n consecutive rows of a snapshot's Qt (n x n, global) into padded shared rows.
__device__ inline void load_Qt_rows(int n, const cd *__restrict__ Qg, cd *__restrict__ Qs, int lane, int nthr) {
    const int lq = ld_qt(n);
    for (int e = lane; e < n * n; e += nthr) {
        int c = e / n, k = e - c * n;
        Qs[c * lq + k] = Qg[e];
    }
}

// The same, also writing re + im of every staged entry to qs (n x n, row stride n).
__device__ inline void load_Qt_rows_sums(int n, const cd *__restrict__ Qg, cd *__restrict__ Qs,
                                         double *__restrict__ qs, int lane, int nthr) {
    const int lq = ld_qt(n);
    for (int e = lane; e < n * n; e += nthr) {
        const int c = e / n, k = e - c * n;
        const cd q = Qg[e];
        Qs[c * lq + k] = q;
        qs[e] = q.x + q.y;
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


// B^(s) (packed upper, m x m) from K = Ut [H1 | G2] (n x 2n, rows of Ks with T's stride)
// and the walker rows Ut, for a snapshot with H1 = Qt^T J Qt, G2 = Qt^T J conj(Qt) (its rows
// [H1^T; G2^T] staged in place of Qt, so that K is formed exactly like T).  With
// W1 = K1 Ut^T = T J T^T and W2 = K2 Ut^H = T J conj(T)^T and the empty rows
// R_j = Re T_j, I_j = -Im T_j of the selection,
//     occupied a < b:             W1[a][b]
//     occupied a, empty mode j:   (a, R_j) = (W1 + W2)[a][j] / 2,  (a, I_j) = i (W1 - W2)[a][j] / 2
//     empty modes j1 <= j2 (al = W1, be = W2 at [j1][j2]):
//         (R, R) = Re(al + be)/2, (R, I) = Im(be - al)/2, (I, R) = -Im(al + be)/2,
//         (I, I) = Re(be - al)/2; within one mode only (R_j, I_j) = Im(be)/2.
// Each sum runs over the non-zero columns of walker row b only: column b and [ne, n) for
// an occupied row in reduced form (red), [b, n) in echelon form, [0, ne) and [b, n) for a
// completion row b >= ne.  Three real products per complex term (Gauss's form, with the
// staged sums Ksum = re + im of K1 and re - im of K2, and Uss = re + im of Ut):
//     K1 u:       Re = p1 - p2, Im = p3 - p1 - p2,   p3 = sum (k1r + k1i)(ur + ui)
//     K2 conj(u) = conj(conj(K2) u): Re = q1 + q2, Im = q1 - q2 - q3,
//                 q3 = sum (k2r - k2i)(ur + ui)   (q1 = sum k2r ur, q2 = sum k2i ui).
// The occupied-empty and empty-empty items share their sums' shape, so they run in one loop
// ordered by completion row b (the ne occupied rows a, then the empty modes up to b):
// neighbouring lanes share their loop bounds.
__device__ inline void build_B_from_K(int n, int ne, bool red, const cd *__restrict__ Uts,
                                      const double *__restrict__ Uss, const cd *__restrict__ Ks,
                                      const double *__restrict__ Ksum,
                                      cd *__restrict__ Bs, const uint16_t *__restrict__ tab, int lane,
                                      int nthr) {
    const int d = n - ne, lu = ld_ut(n), lt = ld_t(n), n2 = 2 * n;
    const int c1 = tri_count(ne);
    for (int e = lane; e < c1; e += nthr) {  // occupied x occupied: W1 alone
        int a, b;
        pair_of(tab, e, a, b);
        const cd *kr = Ks + a * lt, *ur = Uts + b * lu;
        const double *ks = Ksum + a * n2, *us = Uss + b * lu;
        double p1 = 0.0, p2 = 0.0, p3 = 0.0;
        if (red) {
            p1 = kr[b].x * ur[b].x;
            p2 = kr[b].y * ur[b].y;
            p3 = ks[b] * us[b];
        }
        for (int k = red ? ne : b; k < n; ++k) {
            const cd kk = kr[k], u = ur[k];
            p1 = fma(kk.x, u.x, p1);
            p2 = fma(kk.y, u.y, p2);
            p3 = fma(ks[k], us[k], p3);
        }
        Bs[tri_index(a, b)] = cmk(p1 - p2, p3 - p1 - p2);
    }
    const int c2 = ne * d + tri_count(d + 1);
    for (int e = lane; e < c2; e += nthr) {
        // completion row b = ne + jj carries ne + jj + 1 items
        int jj = 0, base = 0;
        while (jj + 1 < d && base + ne + jj + 1 <= e) {
            base += ne + jj + 1;
            ++jj;
        }
        const int i = e - base, b = ne + jj;
        const bool occ = i < ne;
        const int a = i;  // K row: occupied row i (i < ne), or that of empty mode i - ne
        const cd *kr = Ks + a * lt, *ur = Uts + b * lu;
        const double *ks = Ksum + a * n2, *us = Uss + b * lu;
        double p1 = 0.0, p2 = 0.0, p3 = 0.0, q1 = 0.0, q2 = 0.0, q3 = 0.0;
        for (int k = 0; k < ne; ++k) {
            const cd u = ur[k], k1 = kr[k], k2 = kr[n + k];
            p1 = fma(k1.x, u.x, p1);
            p2 = fma(k1.y, u.y, p2);
            p3 = fma(ks[k], us[k], p3);
            q1 = fma(k2.x, u.x, q1);
            q2 = fma(k2.y, u.y, q2);
            q3 = fma(ks[n + k], us[k], q3);
        }
        for (int k = b; k < n; ++k) {
            const cd u = ur[k], k1 = kr[k], k2 = kr[n + k];
            p1 = fma(k1.x, u.x, p1);
            p2 = fma(k1.y, u.y, p2);
            p3 = fma(ks[k], us[k], p3);
            q1 = fma(k2.x, u.x, q1);
            q2 = fma(k2.y, u.y, q2);
            q3 = fma(ks[n + k], us[k], q3);
        }
        const cd w1 = cmk(p1 - p2, p3 - p1 - p2), w2 = cmk(q1 + q2, q1 - q2 - q3);
        if (occ) {
            const cd sp = cadd(w1, w2), dm = csub(w1, w2);
            Bs[tri_index(a, ne + 2 * jj)] = cscale(sp, 0.5);
            Bs[tri_index(a, ne + 2 * jj + 1)] = cmk(-0.5 * dm.y, 0.5 * dm.x);
        } else {
            const int r1 = 2 * (i - ne), r2 = 2 * jj;
            if (r1 < r2) {
                Bs[tri_index(ne + r1, ne + r2)] = cmk(0.5 * (w1.x + w2.x), 0.0);
                Bs[tri_index(ne + r1, ne + r2 + 1)] = cmk(0.5 * (w2.y - w1.y), 0.0);
                Bs[tri_index(ne + r1 + 1, ne + r2)] = cmk(-0.5 * (w1.y + w2.y), 0.0);
                Bs[tri_index(ne + r1 + 1, ne + r2 + 1)] = cmk(0.5 * (w2.x - w1.x), 0.0);
            } else {
                Bs[tri_index(ne + r1, ne + r1 + 1)] = cmk(0.5 * w2.y, 0.0);
            }
        }
    }
}
