// qcs_pairfp64.cuh -- one pair in FP64: for pairs whose fixed-point evaluation would lose its bits.
//
// The fixed-point kernels hold a matrix to 2^-57 of its largest entry.  A walker near a
// computational-basis determinant has entries of very different sizes, and against a signed
// permutation B^(s) can consist of products of the small ones: FP64 keeps their relative
// precision, one scale does not (occupied columns I + 1e-8 A, n = 6, ne = 4: 23 of 64 pairs
// beyond 1e-10 of their own scale).  Such pairs show small pivots (fx_pair_eliminate, kGuard)
// and are evaluated here from the walker's FP64 rows, every node matrix in full with partial
// pivoting.  Rare and bound by the FP64 pipe; one copy, not inlined.
#pragma once
#include "qcs_fixed.cuh"

// T of a signed permutation (codes) or of a dense snapshot (rows Qt), from the rows in global
// memory.
template <class Team>
__device__ __forceinline__ void fp64_T(const Team &tm, int n, const cd *__restrict__ U, const cd *__restrict__ Q,
                                       const uint8_t *__restrict__ code, cd *__restrict__ T) {
    const int n2 = 2 * n, lt = ld_t(n);
#pragma unroll 1
    for (int e = tm.t; e < n * n2; e += Team::NT) {
        const int j = e / n2, c = e - j * n2;
        cd s = cmk(0.0, 0.0);
        if (code) {
            const unsigned q = code[c], ph = q & 3u;
            const cd u = U[j * n + (int)(q >> 2)];
            s = ph == 0u ? u : ph == 1u ? cmk(-u.y, u.x) : ph == 2u ? cmk(-u.x, -u.y) : cmk(u.y, -u.x);
        } else {
#pragma unroll 1
            for (int k = 0; k < n; ++k) cfma(s, U[j * n + k], Q[c * n + k]);
        }
        T[j * lt + c] = s;
    }
}

// sum_k gamma_k pf(B + w_k D), the same value on every thread of the team.  B: tri(m) entries of
// shared memory, T: max(n ld_t(n), tri(m)), GV: m; tm.sync() before the call.
template <class Team>
static __device__ __noinline__ cd fp64_pair_sum(Team tm, int n, int ne, const FxPlan &plan,
                                                const cd *__restrict__ U, const cd *__restrict__ Q,
                                                const uint8_t *__restrict__ code, cd *B, cd *T, cd *GV,
                                                const uint16_t *__restrict__ tab) {
    const int m = 2 * n - ne, d = n - ne, Tm = tri_count(m);
    fp64_T(tm, n, U, Q, code, T);
    tm.sync();
    build_B(n, ne, T, B, tab, tm.t, Team::NT);
    tm.sync();
    cd *N = T;  // the node matrix, once B is formed
    cd S = cmk(0.0, 0.0);
#pragma unroll 1
    for (int k = 0; k < plan.nev; ++k) {
        const cd w = cmk(fx_f64(plan.w[k].x, -58), fx_f64(plan.w[k].y, -58));
        for (int e = tm.t; e < Tm; e += Team::NT) N[e] = B[e];
        tm.sync();
        for (int i = tm.t; i < d; i += Team::NT) {
            cd *x = N + tri_index(ne + 2 * i, ne + 2 * i + 1);
            *x = cadd(*x, w);
        }
        tm.sync();
        cd pf = cmk(fx_f64(plan.g[k].x, plan.ge[k]), fx_f64(plan.g[k].y, plan.ge[k]));
#pragma unroll 1
        for (int r = m; r > 0; r -= 2) {
            // the largest entry of the last row (every warp finds it by itself; only rows before
            // it are written until the barrier after the update)
            const cd *row = N + tri_count(r - 1);
            unsigned key = 0u, at = 0u;
            for (int a = tm.lane; a < r - 1; a += 32) {
                const unsigned h = pivot_key(row[a]);
                if (h > key) {
                    key = h;
                    at = (unsigned)a;
                }
            }
            const unsigned top = __reduce_max_sync(QCS_FULL, key);
            const int P = (int)__reduce_min_sync(QCS_FULL, key == top ? at : 0xffffu);
            const int rv = r - 2;
            pf = cmul(pf, flip_if(row[P], P != rv));
            if (rv == 0 || top == 0u) break;
            const cd inv = cinv(row[P]);
            const int tP = tri_count(P), tL = tri_count(rv);
            // place P takes the index before the last: i reads and writes entries of its own
            for (int i = tm.t; i < rv; i += Team::NT) {
                const int o = i == P ? rv : i;
                const bool lo = o > P;
                cd *a = N + (lo ? tri_count(o) + P : tP + o);
                const cd x = flip_if(*a, lo), y = N[tL + i];
                GV[2 * i] = cmul(row[o], inv);
                GV[2 * i + 1] = x;
                if (i != P) *a = flip_if(y, lo);
            }
            tm.sync();
            for (int u = tm.t; u < tri_count(rv); u += Team::NT) {
                int i, j;
                pair_of(tab, u, i, j);
                cd x = N[u];
                cfma(x, GV[2 * i], GV[2 * j + 1]);
                cfms(x, GV[2 * i + 1], GV[2 * j]);
                N[u] = x;
            }
            tm.sync();
        }
        S = cadd(S, pf);
        tm.sync();  // the node matrix is read to the end
    }
    return S;
}
