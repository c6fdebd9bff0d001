"""fx_sweep (csrc/qcs_fxsweep.cuh) on the CPU: inverses of packed skew-symmetric matrices by sweeps in
fixed point, by one and two warps in different orders between their barriers.  Whole matrices
against numpy; sweeps of a block of one matrix against the block formulas.  Tolerance: a sweep
rounds at 2^-57 of rows scaled to 58 bits and keeps multipliers below 2^3, so each of the m / 2
steps adds at most a few units, amplified by the matrix's condition number: 2^-50 m cond."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import warp_emulation

SOURCE = r"""
template <int NW>
static int sweep(int mc, int stop, int occ, int nb, const long long *X0, int f, int mb, unsigned schedule, double *out,
                 int *perm, int *left) {
    const int T = tri_count(mc);
    std::vector<uint16_t> tab(T);
    build_pair_table(tab.data(), T);
    std::vector<fx2> X(nb * T), pv(nb * mc / 2 + 1);
    std::vector<int> pe(nb * mc / 2 + 1), se(nb * mc), bad(nb);
    std::vector<FxGauss> GV(nb * mc);
    std::vector<int8_t> dl(nb * mc);
    std::vector<uint8_t> pm(nb * mc);
    unsigned scr[4];
    memcpy(X.data(), X0, sizeof(fx2) * nb * T);
    const FxSweepWork wk = {GV.data(), pv.data(), pe.data(), bad.data(), se.data(), dl.data(), pm.data()};
    std::vector<FxSwept> r(32 * NW);
    const bool fin = emu::run(NW, schedule, [&](int t) {
        const FxTeam<NW> tm = {t, t & 31, t >> 5, 1, scr};
        r[t] = fx_sweep(tm, mc, stop, occ != 0, nb, X.data(), f, mb, wk, tab.data());
    });
    if (!fin) return -1;
    for (auto &x : r)
        if (x.f != r[0].f || x.mb != r[0].mb || x.left != r[0].left) return -2;
    *left = r[0].left;
    if (r[0].mb < 0) return 0;
    for (int v = 0; v < nb; ++v)
        for (int j = 0, e = 0; j < mc; ++j)
            for (int i = 0; i < j; ++i, ++e) {
                const int E = -r[0].f - se[v * mc + i] - se[v * mc + j];
                out[2 * (v * T + e)] = std::ldexp((double)X[v * T + e].x, E);
                out[2 * (v * T + e) + 1] = std::ldexp((double)X[v * T + e].y, E);
            }
    for (int e = 0; e < nb * mc; ++e) perm[e] = pm[e];
    return 1;
}
extern "C" int host_sweep(int NW, int mc, int stop, int occ, int nb, const long long *X, int f, int mb, unsigned schedule,
                          double *out, int *perm, int *left) {
    return NW == 1 ? sweep<1>(mc, stop, occ, nb, X, f, mb, schedule, out, perm, left)
                   : sweep<2>(mc, stop, occ, nb, X, f, mb, schedule, out, perm, left);
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    lib = warp_emulation.compile_host(SOURCE, ["qcs_fxsweep.cuh"], str(tmp_path_factory.mktemp("emu")))
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)

    def run(NW, A, stop, occ, schedule):
        """Sweeps the matrices A (nb, mc, mc): (result, perm, left) or None when refused."""
        nb, mc, _ = A.shape
        i, j = np.triu_indices(mc, 1)
        order = np.lexsort((i, j))  # packed: column after column
        i, j = i[order], j[order]
        v = A[:, i, j]
        X = np.stack([np.rint(v.real * 2.0**57), np.rint(v.imag * 2.0**57)], axis=-1).astype(np.int64)
        out, perm, left = np.zeros((nb, len(i), 2)), np.zeros((nb, mc), np.int32), ctypes.c_int()
        r = lib.host_sweep(NW, mc, stop, int(occ), nb, ptr(np.ascontiguousarray(X)), 57, 58, schedule, ptr(out),
                           ptr(perm), ctypes.byref(left))
        assert r >= 0, r  # no deadlock, one outcome on every thread
        if r == 0:
            return None
        R = np.zeros((nb, mc, mc), complex)
        R[:, i, j] = out[..., 0] + 1j * out[..., 1]
        return R - np.transpose(R, (0, 2, 1)), perm, left.value

    return run


def skew(rng, nb, m):
    A = rng.uniform(-1, 1, (nb, m, m)) + 1j * rng.uniform(-1, 1, (nb, m, m))
    A = np.triu(A, 1)
    return A - np.transpose(A, (0, 2, 1))


@pytest.mark.parametrize("NW", [1, 2])
@pytest.mark.parametrize("m,nb", [(2, 1), (4, 3), (6, 2), (8, 4), (16, 3), (24, 1)])
def test_whole_matrices(host, NW, m, nb):
    rng = np.random.default_rng(10 * m + nb)
    A = skew(rng, nb, m)
    first = None
    for schedule in (0, 1, 5):
        r = host(NW, A, 0, False, schedule)
        assert r is not None
        R, perm, _ = r
        for v in range(nb):
            inv = np.zeros((m, m), complex)
            inv[np.ix_(perm[v], perm[v])] = R[v]
            cond = np.linalg.cond(A[v])
            assert np.abs(inv - np.linalg.inv(A[v])).max() <= 2.0**-50 * m * cond * np.abs(inv).max()
        if first is None:
            first = R
        assert np.array_equal(R, first)


@pytest.mark.parametrize("NW", [1, 2])
@pytest.mark.parametrize("d2,ne", [(2, 2), (4, 4), (6, 8), (16, 8), (0, 6), (20, 12)])
def test_a_block(host, NW, d2, ne):
    """[[S, E], [-E^T, P]] to [[S + E P^-1 E^T, E P^-1], [.., P^-1]] on the indices that were swept."""
    rng = np.random.default_rng(100 * d2 + ne)
    A = skew(rng, 1, d2 + ne)
    first = None
    for schedule in (0, 1, 3):
        R, perm, left = host(NW, A, d2, True, schedule)
        keep, p = perm[0][: d2 + left], perm[0][d2 + left:]
        assert sorted(perm[0]) == list(range(d2 + ne)) and list(perm[0][:d2]) == list(range(d2))
        B = A[0]
        Pi = np.linalg.inv(B[np.ix_(p, p)]) if len(p) else np.zeros((0, 0))
        E = B[np.ix_(keep, p)] @ Pi
        S = B[np.ix_(keep, keep)] + E @ B[np.ix_(keep, p)].T
        ref = np.block([[S, E], [-E.T, Pi]])
        cond = np.linalg.cond(B[np.ix_(p, p)]) if len(p) else 1.0
        assert np.abs(R[0] - ref).max() <= 2.0**-50 * (d2 + ne) * cond * max(1.0, np.abs(ref).max())
        if first is None:
            first = R
        assert np.array_equal(R, first)
