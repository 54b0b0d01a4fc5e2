"""Rollout pass with fp32 block scales at the edge of its two forms: batches of one row tile (up to 128 rows) promote that one
alone, longer ones pairs of row tiles; with one block per stage, an even or odd number of stages."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [32, 64, 128])
@pytest.mark.parametrize("T,d", [(1, 384), (127, 256), (128, 384), (128, 512), (129, 384), (300, 256)])
def test_rollout_log_probs_of_one_row_tile_and_of_a_pair(T, d, block):
    import paper_2605_13907_b200 as ais
    V = 1352
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T + block)
    H = torch.randn(T, d, generator=gen, device="cuda").to(torch.bfloat16)
    W = (torch.randn(V, d, generator=gen, device="cuda") * (1.28 / d ** 0.5)).to(torch.bfloat16)
    tokens = torch.randint(0, V, (T,), generator=gen, device="cuda", dtype=torch.int32)
    mask = torch.ones(T, dtype=torch.uint8, device="cuda")
    mask[T // 2] = 0 if T > 1 else 1
    s = ais.AisStep(T, d, V, 1, 1, block, want_grad=False)
    s.forward(H, W, tokens, mask)
    torch.cuda.synchronize()
    assert int(s.status.item()) == 0

    def dequantised(codes, scales, rows):
        x = codes[:, :d].view(torch.float8_e4m3fn).double().reshape(rows, d // block, block)
        return (x * scales[:, :rows].t().double().unsqueeze(2)).reshape(rows, d)

    z = dequantised(s.qH, s.sH, T) @ dequantised(s.qW, s.sW, V).t()
    lse = torch.logsumexp(z, dim=1)
    lp = z.gather(1, tokens.long().unsqueeze(1)).squeeze(1) - lse
    on = mask != 0
    # fp32: up to 16 block sums added to logits of at most 8 (2^-24 of the sum each, twice), a few hundred exponentials added in a
    # row (2^-24 each) and the roundings of exp2, log and lse (2^-20 for 8 <= lse < 16)
    tol = 2.0 ** -16
    assert float((s.lse_roll[:T].double() - lse)[on].abs().max()) <= tol
    assert float((s.lp_roll[:T].double() - lp)[on].abs().max()) <= tol
    assert bool((s.lp_roll[:T][~on] == 0).all())
