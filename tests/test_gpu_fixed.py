"""Fixed-point eliminations (csrc/qcs_fixed.cuh) away from the unit scale of orthogonal
snapshots: Q scaled as a whole, with one large row, and with rows of very different sizes,
evaluated at every node of every snapshot (no parity shortcut holds for such Q), against
the oracle at the FP64 path's 1e-10 of the pair scale; and matrix sizes at the edges of the
elimination (no empty mode, closing blocks of two and four, the largest order one warp or
two take)."""
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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def scaled(kind, Q):
    Q = Q.copy()
    if kind == "eighth":
        Q *= 0.125
    elif kind == "large":
        Q *= 37.0
    elif kind == "one_row":
        Q[:, 3, :] *= 1e3
    elif kind == "graded":
        Q *= 2.0 ** np.linspace(-6, 6, Q.shape[1])[None, :, None]
    return Q


SIZES = [(2, 2), (3, 2), (4, 4), (6, 2), (8, 4), (16, 8), (16, 2), (17, 16), (20, 10)]


# parity-consistent bits: the pair scale of a forbidden pair is rounding noise.  n = 24, ne = 2
# at the unit scale only: the 47 interpolation nodes at |z| = 1 lose nine digits there when
# the covariance is far from norm one, in FP64 eliminations just the same.
@pytest.mark.parametrize("n,ne,kind", [(n, ne, k) for n, ne in SIZES
                                       for k in ("unit", "eighth", "large", "one_row", "graded")] + [(24, 2, "unit")])
def test_scales_and_sizes(ctx, n, ne, kind):
    rng = np.random.default_rng(100 * n + ne)
    W, P = 3, 9
    Q = scaled(kind, synth.haar_orthogonal(rng, 2 * n, P))
    b = synth.parity_consistent_bits(rng, Q)
    Phi = synth.walkers(rng, n, ne, W)
    s = qcs.Snapshots(ctx, dev(Q), dev(b))
    ov, pp = qcs.overlap(ctx, s, dev(Phi), per_pair=True, flags=qcs.QCS_FLAG_ALL_NODES)
    torch.cuda.synchronize()
    assert ctx.sync_status() == 0
    _, opp, sc, _ = orc.overlap(Phi, Q, b, per_pair=True)
    assert np.all(np.abs(pp.cpu().numpy() - opp) <= 1e-10 * sc)


def test_nonfinite_walker_gives_nan(ctx):
    """A walker with a NaN or an infinity gives NaN overlaps, its neighbours their values."""
    rng = np.random.default_rng(5)
    for n, ne in ((8, 4), (16, 8), (20, 10)):
        Q = synth.haar_orthogonal(rng, 2 * n, 20)
        b = synth.parity_consistent_bits(rng, Q)
        Phi = synth.walkers(rng, n, ne, 4)
        good, _, _, _ = orc.overlap(Phi, Q, b, per_pair=True)
        bad = Phi.copy()
        bad[1, 0, 0] = np.nan
        bad[2, 1, 1] = np.inf
        s = qcs.Snapshots(ctx, dev(Q), dev(b))
        ov, _ = qcs.overlap(ctx, s, dev(bad))
        ov = ov.cpu().numpy()
        assert ctx.sync_status() & qcs.QCS_ERR_NONFINITE
        assert np.isnan(ov[1]) and np.isnan(ov[2])
        assert np.allclose(ov[[0, 3]], good[[0, 3]], rtol=1e-10, atol=0)
