"""Quantisers on more rows than 65,535 blocks of a grid dimension cover (2^20 - 16 at sixteen rows per block): bit for bit what
the same rows give in slices, whose codes are checked against the oracle elsewhere."""

import pytest
import torch

pytestmark = pytest.mark.gpu

SLICE = 1 << 18            # rows; a multiple of the 256 rows that the packed scales are grouped by
COLS = 256


@pytest.mark.parametrize("rows", [(1 << 20) + 1, 2_200_000])
@pytest.mark.parametrize("kind", ["per_tensor", "mxfp8", "mxfp4"])
def test_long_batches_quantise_like_their_slices(kind, rows):
    import paper_2605_13907_b200 as ais
    block = {"per_tensor": 0, "mxfp8": ais.FP8_MX32, "mxfp4": ais.FP4_MX32}[kind]
    g = torch.Generator(device="cuda")
    g.manual_seed(rows % 1000)
    x = torch.randn(rows, COLS, generator=g, device="cuda").to(torch.bfloat16)
    x[::SLICE, 0] = 7.0                                     # the maximum of the matrix in every slice
    x.clamp_(-7.0, 7.0)
    codes, scales = ais.quantize_fp8(x, block)
    packed = scales.reshape(-1)
    at = 0
    for r0 in range(0, rows, SLICE):
        part = x[r0:r0 + SLICE]
        c, s = ais.quantize_fp8(part, block)
        assert torch.equal(codes[r0:r0 + SLICE], c), r0
        if block == 0:
            assert packed[0] == s.reshape(-1)[0], r0
        else:
            n = ais.mx_scale_bytes(part.shape[0], COLS)
            assert torch.equal(packed[at:at + n], s), r0
            at += n
    assert block == 0 or at == packed.numel()
