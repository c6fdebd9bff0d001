"""Second moments of the covariance entries on tensor cores (csrc/qcs_rdm.cu): snapshot counts
at the edges of a stage (32), an exact sum (128) and a batch of slices (65536), pair counts
at the edges of the 128 x 64 tiles, covariances away from the unit scale, and snapshots that
are not finite, against plain FP64 torch.

Tolerance 1e-12 K4 s^2 with s the largest covariance entry: each of 128 snapshots' sums is
rounded once at 2^-47 s^2 and the slices at 2^-56, far below 1e-12 of a mean of products of
entries of at most s."""
from __future__ import annotations

from math import comb

import numpy as np
import pytest
import torch

from paper_2506_22408_gb300 import qcs, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return qcs.Context(0)


def reference(Q, b):
    P, N2, _ = Q.shape
    n = N2 // 2
    s = (1 - 2 * b.double())[:, :, None]
    ev, od = Q[:, 0::2, :], Q[:, 1::2, :] * s
    G = ev.transpose(1, 2) @ od
    X = G - G.transpose(1, 2)
    iu = torch.triu_indices(N2, N2, 1, device=Q.device)
    rank = torch.zeros((N2, N2), dtype=torch.long, device=Q.device)
    rank[iu[0], iu[1]] = torch.arange(iu.shape[1], device=Q.device)
    x = X[:, iu[0], iu[1]]
    S2 = x.T @ x / P
    q = torch.combinations(torch.arange(N2, device=Q.device), 4)
    p = lambda i, j: rank[q[:, i], q[:, j]]
    v = S2[p(0, 1), p(2, 3)] - S2[p(0, 2), p(1, 3)] + S2[p(0, 3), p(1, 2)]
    K2, K4 = comb(N2, 2) / n, comb(N2, 4) / comb(n, 2)
    return K2 * X.mean(dim=0), -K4 * v, K2, K4, X.abs().max()


def make(n, P, seed, scale=1.0):
    rng = np.random.default_rng(seed)
    Q = torch.from_numpy(synth.haar_orthogonal(rng, 2 * n, min(P, 700))).cuda()
    Q = Q[torch.arange(P, device="cuda") % Q.shape[0]].contiguous() * scale
    return Q, torch.from_numpy(synth.uniform_bits(rng, n, P)).cuda()


@pytest.mark.parametrize("n,P,scale", [(2, 1, 1.0), (3, 31, 1.0), (6, 32, 1.0), (8, 129, 1.0), (12, 128, 1.0),
                                       (16, 4097, 1.0), (24, 300, 1.0), (4, 65536, 1.0), (5, 66001, 1.0),
                                       (9, 257, 37.0), (16, 500, 2.0**-20), (7, 140, 1e60)])
def test_moments(ctx, n, P, scale):
    Q, b = make(n, P, 10 * n + P, scale)
    out = qcs.shadow_rdm(ctx, qcs.Snapshots(ctx, Q, b))
    torch.cuda.synchronize()
    ctx.sync_status()
    gam2, gam4, K2, K4, s = reference(Q, b)
    assert (out["gam2"] - gam2).abs().max() <= 1e-12 * K2 * s
    assert (out["gam4"] - gam4).abs().max() <= 1e-12 * K4 * s * s


def test_nonfinite_snapshot_reaches_the_same_outputs(ctx):
    Q, b = make(6, 200, 3)
    Q[17, 4, 5] = float("nan")
    out = qcs.shadow_rdm(ctx, qcs.Snapshots(ctx, Q, b))
    torch.cuda.synchronize()
    assert ctx.sync_status() & qcs.QCS_ERR_NONFINITE
    gam2, gam4, K2, K4, _ = reference(Q, b)
    # the covariance's row and column 5 only
    ok = torch.isfinite(gam4)
    assert ok.any() and not ok.all()
    assert torch.equal(torch.isfinite(out["gam4"]), ok)
    assert (out["gam4"][ok] - gam4[ok]).abs().max() <= 1e-12 * K4
