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


def _log_probs_from_codes(s, tokens, T, V, d, block):
    """(lp, lse) in fp64 from the codes and scales that the step holds."""
    def dequantised(codes, scales, rows):
        x = codes[:, :d].view(torch.float8_e4m3fn).double().reshape(rows, d // block, block)
        return (x * scales[:, :rows].t().double().unsqueeze(2)).reshape(rows, d)

    z = dequantised(s.qH, s.sH, T) @ dequantised(s.qW, s.sW, V).t()
    assert float(z.abs().max()) < 8.0
    lse = torch.logsumexp(z, dim=1)
    return z.gather(1, tokens.long().unsqueeze(1)).squeeze(1) - lse, lse


@pytest.mark.parametrize("block", [32, 64, 128])
@pytest.mark.parametrize("T,d,V,ranges", [
    (100, 384, 40008, 0),        # one row tile, three column tiles of three stages per CTA
    (128, 1280, 60000, 0),       # the same with four tiles of ten stages
    (77, 640, 5000, 1),          # one CTA walks all forty tiles
    (300, 384, 40008, 0),        # pairs of row tiles, an odd number of stages
    (900, 640, 20000, 64),       # four pairs x 64 ranges: two units on most CTAs
    (900, 512, 20000, 64),
    (700, 896, 5000, 64),        # seven, eight and nine stages per tile: the two ways in which copies and MMAs of smaller blocks are issued
    (700, 1024, 5000, 64),
    (700, 1152, 5000, 64),
])
def test_rollout_log_probs_over_several_column_tiles(T, d, V, ranges, block):
    """Several column tiles and units per CTA: operand stages, scale slots and accumulator buffers go round more than once, the
    running maximum and sum pass from tile to tile, and whole row tiles without a valid row are stepped over."""
    import paper_2605_13907_b200 as ais
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T + d + block)
    H = torch.randn(T, d, generator=gen, device="cuda").to(torch.bfloat16)
    W = (torch.randn(V, d, generator=gen, device="cuda") * (1.28 / d ** 0.5)).to(torch.bfloat16)
    tokens = torch.randint(0, V, (T,), generator=gen, device="cuda", dtype=torch.int32)
    mask = (torch.rand(T, generator=gen, device="cuda") < 0.9).to(torch.uint8)
    if T == 900:
        mask[256:512] = 0                # a pair of row tiles without a valid row,
        mask[640:768] = 0                # and the second tile of another
    params = ais.default_params(vocab_chunk=-(-V // ranges) if ranges else 0)
    s = ais.AisStep(T, d, V, 1, 1, block, want_grad=False, params=params)
    s.workspace.fill_(0xFF)
    s.forward(H, W, tokens, mask)
    torch.cuda.synchronize()
    assert int(s.status.item()) == 0
    lp, lse = _log_probs_from_codes(s, tokens, T, V, d, block)
    on = mask != 0
    # as above, for d / block block sums added to a logit of at most 8 (2^-24 of the sum each, twice)
    tol = 2.0 ** -16 + d // block * 2.0 ** -20
    assert float((s.lse_roll[:T].double() - lse)[on].abs().max()) <= tol
    assert float((s.lp_roll[:T].double() - lp)[on].abs().max()) <= tol
    assert bool((s.lp_roll[:T][~on] == 0).all())
