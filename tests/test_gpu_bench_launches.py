"""The number of kernels that the benchmark reports for a step: as the library enqueues them."""

import pytest
import torch

import bench
import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,split,kernels", [(2, True, 8),      # quantisers, two passes, merge, loss, gated recompute, dH, its partial sums
                                             (80, False, 8)])   # beyond the merged moments: a launch of their own; no split tail
def test_kernels_of_a_step(P, split, kernels):
    import paper_2605_13907_b200 as ais
    w = workloads.scaled(workloads.WORKLOADS["tiny"], P=P)
    b = workloads.make_batch(w, device="cpu")
    step = ais.AisStep(b.T, w.d, w.V, w.P, w.G, w.block)
    args = [t.cuda() for t in (b.H, b.W, b.tokens, b.mask, b.seq_offsets, b.rewards)]
    assert (b.T <= 592 * 32) == split
    before = step.dH.clone()
    assert bench.kernels_of(lambda: step.step(*args)) == kernels
    torch.cuda.synchronize()
    assert torch.equal(step.dH.view(torch.int16), before.view(torch.int16))        # a capture runs nothing
