"""Pairs of a walker with entries of very different sizes (occupied columns I + eps A) and a signed
permutation, on the CPU: the fixed-point evaluation must hand those whose bits it would lose to
the FP64 one (csrc/qcs_pairfp64.cuh), gathered and dense, one and two warps, and keep every pair
of an ordinary walker.  Reference: the exact value of the same FP64 rows in integers.  Tolerance:
1e-10 of the nodes' magnitudes sum_k |gamma_k pf_k|, or what FP64 roundings of B^(s) allow,
2^-48 sum_ab |d S / d B_ab| sum |terms of B_ab|, where cancellation in B makes that larger, and
2^-96 sum_k |gamma_k| for two roundings at once where every derivative vanishes."""
from __future__ import annotations

import ctypes
from fractions import Fraction

import numpy as np
import pytest

import warp_emulation
from paper_2506_22408_gb300 import qcs, synth

SOURCE = r"""
struct Args {
    int n, ne, NB;
    const cd *U, *Q;
    const uint8_t *code;
    int sparse;
    FxPlan plan;
};
template <int NW>
static int pair(const Args &A, unsigned schedule, double *out) {
    const int n = A.n, ne = A.ne, m = 2 * n - ne, T = tri_count(m), d2 = m - ne, vm = std::max(m, A.NB * d2);
    std::vector<uint16_t> tab(T);
    build_pair_table(tab.data(), T);
    std::vector<int4> Us(n * (n + 1)), Xr(std::max(n * (n + 1), T));
    std::vector<int4> Tr(std::max(std::max(n * ld_t(n), T), A.NB * tri_count(d2)));
    std::vector<fx2> pv(pv_records(vm, A.NB) + ne / 2 + 1);
    std::vector<int> pe(pv.size());
    std::vector<FxGauss> GV(vm);
    unsigned scr[4];
    int8_t rs[2 * QCS_MAX_N];
    const FxWork wk = {GV.data(), pv.data(), pe.data(), pv_records(vm, A.NB)};
    int4 *Ts = Tr.data(), *Qs = Xr.data();
    fx2 *Xs = (fx2 *)Xr.data(), *Ns = (fx2 *)Tr.data();
    std::vector<cd> S(32 * NW);
    std::vector<char> kept(32 * NW);
    const bool fin = emu::run(NW, schedule, [&](int t) {
        const FxTeam<NW> tm = {t, t & 31, t >> 5, 1, scr};
        const unsigned uk = fx_max_key(A.U, n * n, tm.lane);
        const int fU = fx_fraction(uk, 57);
        const bool wide = fx_wide(A.U, n * n, uk, tm.lane);
        fx_stage_rows(n, n * n, A.U, fU, nullptr, Us.data(), t, tm.NT);
        tm.sync();
        int fT = fU - 1, par = 0;
        if (A.code) {
            fx_gather_T(n, Us.data(), A.code, Ts, t, tm.NT);
        } else {
            const int fQ = fx_fraction(fx_balance_rows(n, A.Q, rs, tm.lane), 57);
            unsigned top = 0u;
            tm.sync();
            for (int h = 0; h < 2; ++h) {
                fx_stage_rows(n, n * n, A.Q + h * n * n, fQ, rs + h * n, Qs, t, tm.NT);
                tm.sync();
                top |= fx_build_T(n, ne, Us.data(), Qs, (fx2 *)Ts, h * n, t, tm.NT);
                tm.sync();
            }
            top = tm.or_put(top, par);
            tm.sync();
            const int b = fx_top_bits(tm.or_get(top, par));
            par ^= 1;
            fT = fU + fQ - 58 + 56 - b;
            fx_T_limbs<kFxST>(n, Ts, b, t, tm.NT);
        }
        tm.sync();
        bool shared = true, ok, lost = false;
        do {
            unsigned top = tm.or_put(fx_build_B(n, ne, Ts, Xs, tab.data(), t, tm.NT), par);
            tm.sync();
            const int mb = fx_top_bits(tm.or_get(top, par));
            par ^= 1;
            tm.sync();
            const bool guard = A.code ? wide : A.sparse != 0;
            S[t] = guard ? fx_pair_eliminate<true>(tm, m, ne, shared, A.NB, A.plan, wk, Xs, Ns, 2 * fT - 56, mb,
                                                   tab.data(), ok, &lost)
                         : fx_pair_eliminate(tm, m, ne, shared, A.NB, A.plan, wk, Xs, Ns, 2 * fT - 56, mb, tab.data(), ok);
            shared = false;
            tm.sync();
        } while (!ok && !lost);
        if (lost) {
            S[t] = fp64_pair_sum(tm, n, ne, A.plan, A.U, A.Q, A.code, (cd *)Xs, (cd *)Ns, (cd *)wk.GV, tab.data());
            if (tm.wid) S[t] = cmk(0.0, 0.0);
        }
        kept[t] = !lost;
    });
    if (!fin) return -1;
    for (char k : kept)
        if (k != kept[0]) return -2;
    out[0] = out[1] = 0.0;
    for (int w = 0; w < NW; ++w) {
        out[0] += S[32 * w].x;
        out[1] += S[32 * w].y;
    }
    return kept[0];
}
extern "C" int host_graded(int NW, int n, int ne, int NB, int nev, const double *wg, const double *U, const double *Q,
                           const uint8_t *code, int sparse, unsigned schedule, double *out) {
    qcs_node_plan p;
    memset(&p, 0, sizeof(p));
    p.nev = nev;
    for (int k = 0; k < nev; ++k) {
        p.wnode[k] = cmk(wg[4 * k], wg[4 * k + 1]);
        p.gamma[k] = cmk(wg[4 * k + 2], wg[4 * k + 3]);
    }
    Args A = {n, ne, NB, (const cd *)U, (const cd *)Q, code, sparse};
    fx_make_plan(p, A.plan);
    return NW == 1 ? pair<1>(A, schedule, out) : pair<2>(A, schedule, out);
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    lib = warp_emulation.compile_host(SOURCE, ["qcs_fxcong.cuh", "qcs_pairfp64.cuh"],
                                      str(tmp_path_factory.mktemp("emu")))
    ptr = lambda a: None if a is None else a.ctypes.data_as(ctypes.c_void_p)

    def pair(NW, n, ne, plan, Ut, Qt, code, schedule, sparse=1):
        out = np.zeros(2)
        wg = np.array([[w.real, w.imag, g.real, g.imag] for w, g in plan])
        Ut, Qt = np.ascontiguousarray(Ut), np.ascontiguousarray(Qt)
        r = lib.host_graded(NW, n, ne, min(3, len(plan)), len(plan), ptr(wg), ptr(Ut), ptr(Qt), ptr(code), sparse,
                            schedule, ptr(out))
        return r, complex(*out)

    return pair


def walker_rows(Phi):
    """Orbital rows in the kernels' form: Householder QR, echelon blocks, occupied rows / sqrt 2."""
    n, ne = Phi.shape
    A, U = Phi.astype(complex), np.eye(n, dtype=complex)

    def reflect(M, v, cols):  # M (I - tau v v^H) on the given columns
        M[:, cols] -= np.outer(M[:, cols] @ v, (2.0 / np.vdot(v, v).real) * v.conj())

    for k in range(ne):
        v = np.zeros(n, complex)
        v[k:] = A[k:, k]
        ph = v[k] / abs(v[k]) if v[k] != 0 else 1.0
        v[k] += ph * np.linalg.norm(v)
        A -= np.outer(v, (2.0 / np.vdot(v, v).real) * (v.conj() @ A))
        reflect(U, v, slice(0, n))
    for c0, c1 in ((0, ne), (ne, n)):
        for r in range(c0, c1 - 1):
            y = U[r, r:c1].conj()
            if not np.any(y[1:]):
                continue
            ph = y[0] / abs(y[0]) if y[0] != 0 else 1.0
            v = y.copy()
            v[0] += ph * np.linalg.norm(y)
            reflect(U, v, slice(r, c1))
            U[r, r + 1:c1] = 0.0
    Ut = U.T.copy()
    Ut[:ne] *= 0.70710678118654752440
    return Ut


def snapshot_rows(Q, b):
    s = np.ones(len(Q))
    s[1::2] = 1.0 - 2.0 * (b & 1)
    Qp = Q * s[:, None]
    return Qp[:, 0::2] - 1j * Qp[:, 1::2]


def codes(Qt):
    out = []
    for row in Qt:
        k = int(np.flatnonzero(row)[0])
        out.append(k << 2 | {1: 0, 1j: 1, -1: 2, -1j: 3}[complex(row[k])])
    return np.array(out, np.uint8)


K = 1200  # every number of the reference is an integer times 2^-K


def integer(x):
    v = Fraction(float(x)) * (1 << K)
    assert v.denominator == 1
    return int(v)


def exact(Ut, Qt, n, ne, plan):
    """(S, sum |gamma_k pf_k|, sum_ab |dS/dB_ab| sum |terms of B_ab|) in floats of exact values."""
    d, m = n - ne, 2 * n - ne
    k, c = np.argmax(Qt != 0, axis=1), [complex(x) for x in Qt[np.arange(2 * n), np.argmax(Qt != 0, axis=1)]]
    T = [[None] * (2 * n) for _ in range(n)]
    for j in range(n):
        for col in range(2 * n):
            u = complex(Ut[j, k[col]]) * c[col]  # a unit phase: exact
            T[j][col] = (integer(u.real), integer(u.imag))
    X = []
    for j in range(d):
        X.append([(x, 0) for x, _ in T[ne + j]])
        X.append([(-y, 0) for _, y in T[ne + j]])
    X += [T[x] for x in range(ne)]
    mul = lambda a, b: (a[0] * b[0] - a[1] * b[1], a[0] * b[1] + a[1] * b[0])
    mag = lambda a: abs(a[0]) + abs(a[1])
    B, terms = {}, {}
    for a in range(m):
        for b in range(a + 1, m):
            s, t = [0, 0], 0
            for i in range(n):
                for p, q, sg in ((2 * i, 2 * i + 1, 1), (2 * i + 1, 2 * i, -1)):
                    z = mul(X[a][p], X[b][q])
                    s[0] += sg * z[0]
                    s[1] += sg * z[1]
                    t += mag(X[a][p]) * mag(X[b][q])
            B[a, b] = (s[0] >> K, s[1] >> K)  # entries have far fewer than K fraction bits
            terms[a, b] = Fraction(t, 1 << 2 * K)
    total, size, slope = 0j, 0.0, 0.0
    for w, g in plan:
        wi = (integer(w.real), integer(w.imag))
        A = dict(B)
        for i in range(d):
            z = A[2 * i, 2 * i + 1]
            A[2 * i, 2 * i + 1] = (z[0] + wi[0], z[1] + wi[1])
        memo = {0: (1 << K, 0)}

        def pf(mask):
            if mask not in memo:
                idx = [i for i in range(m) if mask >> i & 1]
                s = [0, 0]
                for j in range(1, len(idx)):
                    z = A[idx[0], idx[j]]
                    if z == (0, 0):
                        continue
                    z = mul(z, pf(mask & ~(1 << idx[0] | 1 << idx[j])))
                    sg = 1 if j % 2 else -1
                    s[0] += sg * (z[0] >> K)
                    s[1] += sg * (z[1] >> K)
                memo[mask] = tuple(s)
            return memo[mask]

        full = (1 << m) - 1
        value = lambda z: complex(Fraction(z[0], 1 << K), Fraction(z[1], 1 << K))
        v = value(pf(full))
        total += g * v
        size += abs(g * v)
        for (a, b), t in terms.items():
            slope += abs(g) * abs(value(pf(full & ~(1 << a | 1 << b)))) * float(t)
        slope += abs(g) * 2.0**-48
    return total, size, slope


def draw(n, ne, eps, P, seed):
    rng = np.random.default_rng(seed)
    Q = synth.signed_permutation(rng, 2 * n, P)
    b = synth.parity_consistent_bits(rng, Q)
    Phi = np.eye(n)[:, :ne] + eps * (rng.standard_normal((n, ne)) + 1j * rng.standard_normal((n, ne)))
    return walker_rows(Phi), [snapshot_rows(q, x) for q, x in zip(Q, b)]


@pytest.mark.parametrize("n,ne", [(4, 2), (4, 4), (5, 2), (6, 4)])
@pytest.mark.parametrize("eps", [1e-2, 1e-3, 1e-4, 1e-6, 1e-8, 1e-12, 1e-20])
def test_graded_walkers(host, n, ne, eps):
    plan = list(zip(*qcs.node_plan(n, ne)))
    Ut, snaps = draw(n, ne, eps, 10, 17 * n + ne)
    handed = 0
    for i, Qt in enumerate(snaps):
        ref, size, slope = exact(Ut, Qt, n, ne, plan)
        tol = 1e-10 * size + 2.0**-48 * slope
        code = codes(Qt)
        for NW, c, schedule in ((1, code, 0), (1, None, 0), (2, code, i % 2), (2, None, 3)):
            kept, S = host(NW, n, ne, plan, Ut, Qt, c, schedule)
            assert kept in (0, 1), kept
            assert abs(S - ref) <= tol, (i, NW, c is None, kept, abs(S - ref), tol)
            handed += not kept
    if eps <= 1e-8 and ne < n:
        assert handed  # the guard is what keeps them


@pytest.mark.parametrize("n,ne", [(4, 2), (6, 2), (6, 4)])
def test_basis_determinants_need_no_second_evaluation(host, n, ne):
    """Exact zeros of gathered pairs are exact: no pair of a basis determinant is handed over."""
    plan = list(zip(*qcs.node_plan(n, ne)))
    Ut, snaps = draw(n, ne, 0.0, 12, n)
    for Qt in snaps:
        ref, size, slope = exact(Ut, Qt, n, ne, plan)
        kept, S = host(1, n, ne, plan, Ut, Qt, codes(Qt), 0)
        assert kept == 1 and abs(S - ref) <= 1e-10 * size + 2.0**-48 * slope


@pytest.mark.parametrize("n,ne", [(6, 4), (8, 4), (8, 6), (10, 4)])
def test_ordinary_pairs_stay_in_fixed_point(host, n, ne):
    rng = np.random.default_rng(n)
    plan = list(zip(*qcs.node_plan(n, ne)))
    Q = synth.haar_orthogonal(rng, 2 * n, 12)
    b = synth.parity_consistent_bits(rng, Q)
    for q, x, Phi in zip(Q, b, synth.walkers(rng, n, ne, 12)):
        kept, _ = host(1, n, ne, plan, walker_rows(Phi), snapshot_rows(q, x), None, 0, sparse=0)
        assert kept == 1
