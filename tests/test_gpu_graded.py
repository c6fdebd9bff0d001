"""Walkers near a computational-basis determinant (occupied columns I + eps A) against signed
permutations and the same with one 45-degree rotation (a dense snapshot): every pair of the
FP64 ALU path within 1e-10 of its own scale sum_k |gamma_k pf_k|, or within what FP64
roundings of B^(s) allow, 2^-48 sum_ab |dS/dB_ab| sum |terms of B_ab| (and 2^-96 of the scale of
the weights where every derivative vanishes).  The reference is the estimator from the walker in
128-bit numbers."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2506_22408_gb300 import qcs, synth

pytestmark = pytest.mark.gpu
L, CL = np.longdouble, np.clongdouble


@pytest.fixture(scope="module")
def ctx():
    if np.finfo(L).nmant < 100:
        pytest.skip("needs a 128-bit long double (Arm)")
    return qcs.Context(0)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def pfaffian(A):
    A, pf = A.copy(), CL(1)
    for r in range(len(A), 0, -2):
        p = int(np.argmax(np.abs(A[: r - 1, r - 1])))
        if p != r - 2:
            A[[p, r - 2]] = A[[r - 2, p]]
            A[:, [p, r - 2]] = A[:, [r - 2, p]]
            pf = -pf
        piv = A[r - 2, r - 1]
        pf = pf * piv
        if piv == 0:
            return CL(0)
        g, v = A[: r - 2, r - 1] / piv, A[: r - 2, r - 2].copy()
        A[: r - 2, : r - 2] += np.outer(g, v) - np.outer(v, g)
    return pf


def orbitals(Phi):
    """Complete Householder QR: U (occupied columns first) and det R."""
    n, ne = Phi.shape
    A, U, det = Phi.astype(CL), np.eye(n, dtype=CL), CL(1)
    for k in range(ne):
        v = A[:, k].copy()
        v[:k] = 0
        norm = np.sqrt((np.abs(v) ** 2).sum())
        al = -(v[k] / np.abs(v[k])) * norm
        v[k] -= al
        tau = L(2) / (np.abs(v) ** 2).sum()
        A -= tau * np.outer(v, v.conj() @ A)
        U -= tau * np.outer(U @ v, v.conj())
        det *= al
    return U, det


def reference(U, det, Q, b, n, ne, plan):
    """o_p, its scale and its tolerance."""
    s = np.ones(2 * n, dtype=L)
    s[1::2] = 1 - 2 * (b.astype(int) & 1)
    Qp = Q.astype(L) * s[:, None]
    Ut = U.T.copy()
    Ut[:ne] /= np.sqrt(L(2))
    T = Ut @ (Qp[:, 0::2] - 1j * Qp[:, 1::2]).T
    d, m = n - ne, 2 * n - ne
    X = np.zeros((m, 2 * n), dtype=CL)
    X[:ne] = T[:ne]
    X[ne::2], X[ne + 1 :: 2] = T[ne:].real, -T[ne:].imag
    B = X[:, 0::2] @ X[:, 1::2].T - X[:, 1::2] @ X[:, 0::2].T
    aX = np.abs(X)
    terms = aX[:, 0::2] @ aX[:, 1::2].T + aX[:, 1::2] @ aX[:, 0::2].T
    D = np.zeros((m, m))
    for i in range(d):
        D[ne + 2 * i, ne + 2 * i + 1], D[ne + 2 * i + 1, ne + 2 * i] = 1, -1
    S, size, slope = CL(0), L(0), L(0)
    for w, g in plan:
        A = B + CL(w) * D
        v = pfaffian(A)
        S, size = S + CL(g) * v, size + abs(g) * np.abs(v)
        for a in range(m):  # a Pfaffian is affine in every entry
            for c in range(a + 1, m):
                E = A.copy()
                E[a, c] += 1
                E[c, a] -= 1
                slope += abs(g) * np.abs(pfaffian(E) - v) * terms[a, c]
        slope += abs(g) * L(2) ** -48
    pref = 2 * det * CL(1j) ** (ne // 2) / L(2) ** (n - ne // 2)
    return pref * S, np.abs(pref) * (L(10) ** -10 * size + L(2) ** -48 * slope)


def draw(n, ne, eps, P, dense, seed):
    rng = np.random.default_rng(seed)
    Q = synth.signed_permutation(rng, 2 * n, P)
    if dense:
        r = np.eye(2 * n)
        r[0, 0] = r[3, 3] = r[0, 3] = np.sqrt(0.5)
        r[3, 0] = -r[0, 3]
        Q = Q @ r
    b = synth.parity_consistent_bits(rng, Q)
    Phi = np.eye(n)[:, :ne] + eps * (rng.standard_normal((n, ne)) + 1j * rng.standard_normal((n, ne)))
    return Q, b, np.ascontiguousarray(Phi[None])


# one warp per pair, and two above 16 modes
@pytest.mark.parametrize("n,ne,P", [(6, 4, 40), (6, 2, 30), (12, 10, 12), (17, 16, 10), (18, 16, 8)])
@pytest.mark.parametrize("eps", [1e-3, 1e-6, 1e-8])
@pytest.mark.parametrize("dense", [False, True])
def test_every_pair_within_its_own_scale(ctx, n, ne, P, eps, dense):
    Q, b, Phi = draw(n, ne, eps, P, dense, 7 * n + ne)
    s = qcs.Snapshots(ctx, dev(Q), dev(b))
    _, pp = qcs.overlap(ctx, s, dev(Phi), per_pair=True, flags=qcs.QCS_FLAG_FP64_ALU)
    torch.cuda.synchronize()
    assert ctx.sync_status() == 0
    pp = pp.cpu().numpy()[0]
    U, det = orbitals(Phi[0])
    plan = list(zip(*qcs.node_plan(n, ne)))
    for p in range(P):
        ref, tol = reference(U, det, Q[p], b[p], n, ne, plan)
        assert np.abs(pp[p] - ref) <= tol, (p, pp[p], ref, tol)


def test_other_calls_on_the_same_path(ctx):
    """A set of one snapshot makes the mean the pair's value: batched and allocation-free calls."""
    n, ne, P = 6, 4, 12
    Q, b, Phi = draw(n, ne, 1e-8, P, False, 5)
    s = qcs.Snapshots(ctx, dev(Q), dev(b))
    _, pp = qcs.overlap(ctx, s, dev(Phi), per_pair=True)
    pp = pp[0]
    for p in range(P):
        one = qcs.Snapshots(ctx, dev(Q[p : p + 1]), dev(b[p : p + 1]))
        got = qcs.overlap_batched(ctx, [(one, dev(Phi)), (one, dev(Phi))])
        out = torch.zeros(1, dtype=torch.complex128, device="cuda")
        qcs.overlap_noalloc(dev(Q[p : p + 1]), dev(b[p : p + 1]), dev(Phi), out)
        torch.cuda.synchronize()
        for v in (got[0][0], got[1][0], out[0]):
            assert abs(complex(v) - complex(pp[p])) <= 1e-13 * abs(complex(pp[p]))
    assert ctx.sync_status() == 0
