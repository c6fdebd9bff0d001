"""Local energies at sizes where the fixed-point products (csrc/qcs_energy.cu) change shape:
five and more node matrices per round, no empty mode, one mode pair, the node plans that
need several rounds, operators of very different magnitude (each has its own scale).

Tolerance: products of 56-bit numbers with one scale per matrix err by about 2^-56 of
the scales per term, so the sums are as accurate as FP64 ones up to the spread of the
entries: 1e-8 relative to max(1, |value|), times the operators' scale squared (e2) or not
(e1), as for the other local-energy comparisons with the oracle.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle.oracle as orc
from paper_2506_22408_gb300 import qcs, synth

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n,ne,W,P,nchol,flags,scale", [(2, 2, 2, 9, 2, 0, 1.0), (6, 6, 2, 9, 2, 0, 1.0),
                                                        (9, 4, 2, 7, 3, 0, 1.0), (18, 2, 1, 5, 2, 0, 1.0),
                                                        (11, 2, 1, 5, 2, qcs.QCS_FLAG_ALL_NODES, 1.0),
                                                        (8, 4, 2, 9, 2, 0, 1e6), (8, 4, 2, 9, 2, 0, 1e-6)])
def test_matches_oracle(n, ne, W, P, nchol, flags, scale):
    ctx = qcs.Context(0)
    rng = np.random.default_rng(90 + 31 * n + ne)
    Q = synth.haar_orthogonal(rng, 2 * n, P)
    b = synth.parity_consistent_bits(rng, Q)
    Phi = synth.walkers(rng, n, ne, W)
    L = scale * (rng.standard_normal((nchol, n, n)) + 0.3j * rng.standard_normal((nchol, n, n)))
    L[0] *= 1e-3
    h = synth.cholesky_vectors(rng, n, 1)[0].astype(complex)
    s = qcs.Snapshots(ctx, dev(Q), dev(b))
    _, e1, e2 = qcs.local_energy(ctx, s, dev(Phi), dev(L), dev(h), flags=flags)
    torch.cuda.synchronize()
    assert ctx.sync_status() == 0
    _, o1, o2 = orc.local_energy(Phi, Q, b, L, h=h)
    for got, ref, s2 in ((e1, o1, 1.0), (e2, o2, scale * scale)):
        got = got.cpu().numpy()
        assert np.all(np.abs(got - ref) <= 1e-8 * np.maximum(s2, np.abs(ref))), (got, ref)
