"""Local-energy terms of walkers near a basis determinant (occupied columns I + eps A) against signed
permutations: node matrices with small pivots, whose traces are differences of large terms,
within the local energy's 1e-9 of the oracle."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle.oracle as orc
from paper_2506_22408_gb300 import qcs, synth

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n,ne,P", [(8, 4, 40), (12, 6, 40), (10, 4, 200)])
@pytest.mark.parametrize("eps", [0.1, 3e-4, 1e-4])
def test_terms_match_oracle(n, ne, P, eps):
    rng = np.random.default_rng(3)
    Q = synth.signed_permutation(rng, 2 * n, P)
    b = synth.parity_consistent_bits(rng, Q)
    A = rng.standard_normal((n, ne)) + 1j * rng.standard_normal((n, ne))
    L = synth.cholesky_vectors(rng, n, 3).astype(complex)
    h = synth.cholesky_vectors(rng, n, 1)[0].astype(complex)
    Phi = (np.eye(n)[:, :ne] + eps * A)[None]
    ctx = qcs.Context(0)
    got = qcs.local_energy(ctx, qcs.Snapshots(ctx, dev(Q), dev(b)), dev(Phi), dev(L), dev(h))
    torch.cuda.synchronize()
    assert ctx.sync_status() == 0
    ref = orc.local_energy(Phi, Q, b, L, h)
    for x, y in zip(got, ref[:3]):
        assert abs(complex(x[0]) - complex(y[0])) <= 1e-9 * abs(complex(y[0]))
