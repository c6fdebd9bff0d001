"""fx_pair_eliminate (csrc/qcs_fixed.cuh) on the CPU, one and two warps per pair, under different
orders in which the warps run between their barriers: the value must not depend on it (two
warps that disagree about a pivot also wait for each other at different barriers).  The case
that tells them apart: the pivot already stands last, and rewriting column p negates an entry
just below it, whose truncated magnitude then ties with the pivot's."""
from __future__ import annotations

import ctypes
from fractions import Fraction

import numpy as np
import pytest

import warp_emulation

SOURCE = r"""
template <int NW>
static int pair(int m, int ne, int shared, int NB, const FxPlan &plan, const long long *X0, int f, int mb,
                unsigned schedule, double *out) {
    const int T = tri_count(m), d2 = m - ne, vm = std::max(m, NB * d2), Tn = tri_count(d2);
    std::vector<uint16_t> tab(T);
    build_pair_table(tab.data(), T);
    std::vector<fx2> X(T), Ns(std::max(T, NB * Tn)), pv(pv_records(vm, NB) + ne / 2 + 1);
    std::vector<int> pe(pv.size());
    std::vector<FxGauss> GV(vm);
    unsigned scr[4];
    memcpy(X.data(), X0, sizeof(fx2) * T);
    const FxWork wk = {GV.data(), pv.data(), pe.data(), pv_records(vm, NB)};
    std::vector<cd> S(32 * NW);
    std::vector<char> oks(32 * NW);
    const bool fin = emu::run(NW, schedule, [&](int t) {
        const FxTeam<NW> tm = {t, t & 31, t >> 5, 1, scr};
        bool ok;
        S[t] = fx_pair_eliminate(tm, m, ne, shared != 0, NB, plan, wk, X.data(), Ns.data(), f, mb, tab.data(), ok);
        oks[t] = ok;
    });
    if (!fin) return -1;
    for (char k : oks)
        if (k != oks[0]) return -2;
    out[0] = out[1] = 0.0;
    for (int w = 0; w < NW; ++w) {
        out[0] += S[32 * w].x;
        out[1] += S[32 * w].y;
    }
    return oks[0];
}
extern "C" int host_pair(int NW, int m, int ne, int shared, int NB, int nev, const double *wg, const long long *X, int f,
                         int mb, unsigned schedule, double *out) {
    qcs_node_plan p;
    memset(&p, 0, sizeof(p));
    p.nev = nev;
    for (int k = 0; k < nev; ++k) {
        p.wnode[k] = cmk(wg[4 * k], wg[4 * k + 1]);
        p.gamma[k] = cmk(wg[4 * k + 2], wg[4 * k + 3]);
    }
    FxPlan q;
    fx_make_plan(p, q);
    return NW == 1 ? pair<1>(m, ne, shared, NB, q, X, f, mb, schedule, out)
                   : pair<2>(m, ne, shared, NB, q, X, f, mb, schedule, out);
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    lib = warp_emulation.compile_host(SOURCE, ["qcs_fixed.cuh"], str(tmp_path_factory.mktemp("emu")))

    def pair(NW, m, ne, shared, NB, plan, X, f, mb, schedule):
        out = np.zeros(2)
        wg = np.array([[w.real, w.imag, g.real, g.imag] for w, g in plan])
        X = np.ascontiguousarray(X, np.int64)
        r = lib.host_pair(NW, m, ne, int(shared), NB, len(plan), wg.ctypes.data_as(ctypes.c_void_p),
                          X.ctypes.data_as(ctypes.c_void_p), f, mb, schedule, out.ctypes.data_as(ctypes.c_void_p))
        return r, complex(*out)

    return pair


def pfaffian(A):
    """By expansion along the last pivot (Parlett-Reid with partial pivoting)."""
    A, pf = A.copy(), 1.0 + 0j
    while len(A):
        r = len(A)
        p = int(np.argmax(np.abs(A[: r - 1, r - 1])))
        if p != r - 2:
            A[[p, r - 2]] = A[[r - 2, p]]
            A[:, [p, r - 2]] = A[:, [r - 2, p]]
            pf = -pf
        piv = A[r - 2, r - 1]
        pf *= piv
        if piv == 0:
            return 0j
        g, v = A[: r - 2, r - 1] / piv, A[: r - 2, r - 2]
        A = A[: r - 2, : r - 2] + np.outer(g, v) - np.outer(v, g)
    return pf


def unpack(X, m, f):
    A = np.zeros((m, m), complex)
    t = 0
    for j in range(m):
        for i in range(j):
            A[i, j] = complex(*(np.asarray(X[t], float) * 2.0**-f))
            A[j, i] = -A[i, j]
            t += 1
    return A


def reference(X, m, ne, plan, f):
    B, D = unpack(X, m, f), np.zeros((m, m))
    for i in range(0, m - ne, 2):
        D[i, i + 1], D[i + 1, i] = 1.0, -1.0
    terms = [g * pfaffian(B + w * D) for w, g in plan]
    return sum(terms), sum(map(abs, terms))


PLAN = [(np.exp(0.3j), 1.25 + 0j), (np.exp(1.1j), 0.5 - 0.25j), (np.exp(2.0j), -2.0 + 0j)]


def near_tie(d2, ne, rng):
    """The last row's entry (d2, m - 1) is the pivot; the next row's entry (d2 + 1, m - 2) is one
    unit below it, so that its truncated key is one smaller, and its negative's is the same."""
    m = d2 + ne
    X = rng.integers(-(1 << 54), 1 << 54, (m * (m - 1) // 2, 2))
    tri = lambda i, j: j * (j - 1) // 2 + i
    X[tri(d2, m - 1)] = (1 << 57, 0)
    X[tri(d2 + 1, m - 2)] = ((1 << 57) - 1, 0)
    return X


@pytest.mark.parametrize("NW", [1, 2])
@pytest.mark.parametrize("d2,ne", [(2, 4), (6, 6), (16, 8), (24, 12)])
def test_a_pivot_that_stands_last(host, NW, d2, ne):
    rng = np.random.default_rng(d2)
    X, m = near_tie(d2, ne, rng), d2 + ne
    ref, scale = reference(X, m, ne, PLAN, 57)
    first = None
    for schedule in (0, 1, 2, 7, 11):
        r, S = host(NW, m, ne, True, 3, PLAN, X, 57, 58, schedule)
        assert r == 1, (schedule, r)  # no deadlock, one outcome on every thread
        assert abs(S - ref) <= 1e-12 * scale
        first = S if first is None else first
        assert S == first


@pytest.mark.parametrize("NW", [1, 2])
@pytest.mark.parametrize("d2,ne,shared", [(0, 8, True), (4, 2, True), (10, 10, True), (12, 6, False), (20, 14, True)])
@pytest.mark.parametrize("kind", ["random", "signs"])
def test_schedules_agree(host, NW, d2, ne, shared, kind):
    """Random entries, and entries of one magnitude (ties in every step)."""
    rng = np.random.default_rng(7 * d2 + ne)
    m = d2 + ne
    T = m * (m - 1) // 2
    if kind == "random":
        X = rng.integers(-(1 << 57), 1 << 57, (T, 2))
    else:
        X = rng.choice([-1, 1], (T, 2)) * ((1 << 56) - 1)
    ref, scale = reference(X, m, ne, PLAN, 57)
    results = [host(NW, m, ne, shared, 2, PLAN, X, 57, 58, s) for s in (0, 1, 3)]
    assert all(x == results[0] for x in results) and results[0][0] >= 0
    if results[0][0] == 1:
        assert abs(results[0][1] - ref) <= 1e-10 * scale


def exact_pf4(X, w, f):
    """Exact pf of the 4 x 4 matrix X 2^-f + w D (D pairs (0, 1) and (2, 3))."""
    z = [(Fraction(int(x), 1 << f), Fraction(int(y), 1 << f)) for x, y in X]  # 01, 02, 12, 03, 13, 23
    wd = (Fraction(w.real), Fraction(w.imag))
    add = lambda a, b: (a[0] + b[0], a[1] + b[1])
    mul = lambda a, b: (a[0] * b[0] - a[1] * b[1], a[0] * b[1] + a[1] * b[0])
    p, q, r = mul(add(z[0], wd), add(z[5], wd)), mul(z[1], z[4]), mul(z[3], z[2])
    return p[0] - q[0] + r[0], p[1] - q[1] + r[1]


@pytest.mark.parametrize("bits", [52, 54, 57])
def test_a_complement_of_four_keeps_its_bits(host, bits):
    """Without an occupied index or an update, whatever bits B arrives with: entries below two
    in modulus are held to 2^-57 (half a unit lost in the closing shift, w to 2^-59), which a
    product of two turns into at most 4 * 2 * 2^-58 for its part, its dropped limb product and
    rounding into as much again; three products: 6 2^-55.  The value's own rounding to FP64 and
    the product with gamma (normalised to 60 bits) add 2^-53 + 2^-56 of its modulus."""
    rng = np.random.default_rng(bits)
    for _ in range(40):
        X = rng.integers(-(1 << bits), 1 << bits, (6, 2))
        X[rng.integers(6)] = ((1 << bits) - 1, 0)
        w = np.exp(2j * np.pi * rng.random())
        r, S = host(1, 4, 0, True, 1, [(w, 1.0 + 0j)], X, bits, bits, 0)
        ex = exact_pf4(X, w, bits)
        assert r == 1
        tol = Fraction(6, 1 << 55) + Fraction(abs(S)) * Fraction(9, 1 << 56)
        assert max(abs(Fraction(S.real) - ex[0]), abs(Fraction(S.imag) - ex[1])) <= tol
