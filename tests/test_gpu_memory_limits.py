"""Calls that work in batches (tensor-core overlaps, RDMs) when the allocator refuses large
blocks: the same values from smaller batches, a repeated call that asks for nothing (also while
a graph is captured), an error only when the smallest batch is refused too, and working calls
after it.  Values agree to the order of the batches' sums: 1e-13 of the mean magnitude."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2506_22408_gb300 import qcs, synth

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


class CappedContext(qcs.Context):
    """A context whose allocator gives blocks of at most `cap` bytes."""

    def __init__(self):
        super().__init__(0)
        self.cap, self.asked = 1 << 60, []

        def _alloc(nbytes, stream, user):
            self.asked.append(int(nbytes))
            if nbytes > self.cap:
                return None
            return torch.cuda.caching_allocator_alloc(int(nbytes), device=self.device, stream=int(stream or 0))

        def _free(ptr, nbytes, stream, user):
            torch.cuda.caching_allocator_delete(ptr)

        cbs = (qcs._ALLOC_FN(_alloc), qcs._FREE_FN(_free))
        self.check(self.lib.qcs_set_allocator(self.h, cbs[0], cbs[1], None))
        self._allocator_callbacks = cbs


def make(n, ne, W, P):
    rng = np.random.default_rng(10 * n + ne)
    Q = synth.haar_orthogonal(rng, 2 * n, P)
    return dev(Q), dev(synth.parity_consistent_bits(rng, Q)), dev(synth.walkers(rng, n, ne, W))


# the workspace with the largest batch takes 126, 126, 157 and 6 MB
@pytest.mark.parametrize("n,ne,W,P,cap", [(16, 8, 40, 700, 64 << 20), (16, 8, 40, 700, 9 << 20), (16, 2, 23, 901, 3 << 20),
                                          (9, 4, 11, 333, 1 << 20)])
def test_overlaps_in_smaller_batches(n, ne, W, P, cap):
    Q, b, Phi = make(n, ne, W, P)
    plain = qcs.Context(0)
    ref, rpp = qcs.overlap(plain, qcs.Snapshots(plain, Q, b), Phi, per_pair=True, flags=qcs.QCS_FLAG_FP64_TC)
    ctx = CappedContext()
    s = qcs.Snapshots(ctx, Q, b)
    if n < 16:  # the set's records, formed on first use, are not the workspace
        qcs.overlap(ctx, s, Phi[:1], flags=qcs.QCS_FLAG_FP64_TC)
    ctx.cap = cap
    run = lambda: qcs.overlap(ctx, s, Phi, per_pair=True, flags=qcs.QCS_FLAG_FP64_TC)
    ov, pp = run()
    torch.cuda.synchronize()
    assert ctx.sync_status() == 0
    assert max(ctx.asked) > cap >= ctx.workspace_bytes()
    assert torch.equal(pp, rpp)  # a pair's value does not depend on its batch
    tol = 1e-13 * rpp.abs().mean(dim=1)
    assert bool(((ov - ref).abs() <= tol).all())
    asked = len(ctx.asked)
    again, _ = run()
    assert torch.equal(again, ov) and len(ctx.asked) == asked
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        run()
    torch.cuda.current_stream().wait_stream(side)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out, _ = run()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ov) and len(ctx.asked) == asked and ctx.sync_status() == 0


@pytest.mark.parametrize("n,P,cap", [(16, 3000, 40 << 20), (16, 3000, 16 << 20), (7, 1111, 1500 << 10)])
def test_rdms_in_smaller_batches(n, P, cap):
    Q, b, _ = make(n, 2, 1, P)
    plain = qcs.Context(0)
    ref = qcs.shadow_rdm(plain, qcs.Snapshots(plain, Q, b))
    ctx = CappedContext()
    s = qcs.Snapshots(ctx, Q, b)
    ctx.cap = cap
    got = qcs.shadow_rdm(ctx, s)
    torch.cuda.synchronize()
    assert ctx.sync_status() == 0
    assert max(ctx.asked) > cap >= ctx.workspace_bytes()
    names = list(ref) if isinstance(ref, dict) else range(len(ref))
    for k in names:
        # a sum of moments is exact per split; splits are rounded once each
        assert bool(((got[k] - ref[k]).abs() <= 1e-13 * ref[k].abs().max()).all())
    asked = len(ctx.asked)
    qcs.shadow_rdm(ctx, s)
    assert len(ctx.asked) == asked


def test_refused_to_the_last():
    """Not even the smallest batch: QCS_ERR_CUDA, and the context works once it gets memory."""
    Q, b, Phi = make(16, 8, 6, 90)
    ctx = CappedContext()
    s = qcs.Snapshots(ctx, Q, b)
    ref, _ = qcs.overlap(ctx, s, Phi)
    ctx.use_cuda_malloc()
    ctx = CappedContext()
    s = qcs.Snapshots(ctx, Q, b)
    ctx.cap = 10000
    for call in (lambda: qcs.overlap(ctx, s, Phi), lambda: qcs.shadow_rdm(ctx, s)):
        with pytest.raises(qcs.QCSError):
            call()
    ctx.cap = 1 << 60
    ov, _ = qcs.overlap(ctx, s, Phi)
    torch.cuda.synchronize()
    assert ctx.sync_status() == 0
    assert bool(((ov - ref).abs() <= 1e-13 * ref.abs().max()).all())
