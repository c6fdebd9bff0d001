"""Gradients from the fixed-point sweeps (csrc/qcs_fxsweep.cuh, csrc/qcs_grad.cu) against the
CPU oracle where the sweeps change shape: one and many occupied pairs, one and many empty
modes, no empty mode, node matrices in several rounds, several pairs per tile, the largest
mode count, and pairs whose occupied pivots are small (structured walkers, left to the node
matrices) or vanish (FP64 path).

Tolerance, per walker: a sweep of m/2 steps rounds each entry at 2^-57 of its row's scale per
step, and an inverse assembled from the blocks loses at most twice the 4 bits by which a
multiplier may exceed one: 2^-57 m 2^8 < 1e-13 for m <= 46.  Random pairs at these counts have
inverses up to 1e3 of the node matrices' scale, which FP64 inputs multiply: 1e-10 of the
largest gradient entry, plus 1e-11 of the mean pair scale for entries that cancel.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle.oracle as orc
from paper_2506_22408_gb300 import qcs, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return qcs.Context(0)


def _compare(ctx, Q, b, Phi):
    s = qcs.Snapshots(ctx, torch.from_numpy(Q).cuda(), torch.from_numpy(b).cuda())
    ov, g = qcs.overlap_grad(ctx, s, torch.from_numpy(Phi).cuda())
    torch.cuda.synchronize()
    assert ctx.sync_status() == 0
    oo, og, _ = orc.overlap_grad(Phi, Q, b)
    _, _, sc, _ = orc.overlap(Phi, Q, b, per_pair=True)
    for w in range(Phi.shape[0]):
        tol = 1e-10 * np.abs(og[w]).max() + 1e-11 * sc[w].mean()
        assert np.abs(g[w].cpu().numpy() - og[w]).max() <= tol
        assert abs(ov[w].item() - oo[w]) <= 1e-11 * sc[w].mean()


@pytest.mark.parametrize("n,ne,W,P", [(2, 2, 3, 9), (3, 2, 3, 33), (5, 4, 2, 21), (9, 2, 3, 21), (11, 8, 2, 19),
                                      (14, 14, 2, 7), (17, 6, 2, 11), (20, 10, 1, 9), (24, 4, 1, 5), (24, 14, 1, 5)])
def test_sizes(ctx, n, ne, W, P):
    rng = np.random.default_rng(500 + 31 * n + ne)
    Q = synth.haar_orthogonal(rng, 2 * n, P)
    b = synth.parity_consistent_bits(rng, Q)
    _compare(ctx, Q, b, synth.walkers(rng, n, ne, W))


@pytest.mark.parametrize("n,ne,eps", [(8, 4, 1e-2), (8, 4, 1e-5), (12, 6, 0.0)])
def test_weak_occupied_block(ctx, n, ne, eps):
    """Snapshots near the identity: the walker's occupied rows then couple weakly."""
    rng = np.random.default_rng(7 + n)
    P = 12
    A = rng.standard_normal((P, 2 * n, 2 * n))
    Q = np.linalg.qr(np.eye(2 * n) + eps * (A - A.transpose(0, 2, 1)))[0]
    Q = np.ascontiguousarray(Q @ synth.haar_orthogonal(rng, 2 * n, 1))
    b = synth.parity_consistent_bits(rng, Q)
    _compare(ctx, Q, b, synth.walkers(rng, n, ne, 3))
