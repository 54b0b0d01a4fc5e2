"""The batch moments as part of the merge of the log-probs, which a step takes up to 18,944 rows (592 blocks of 32)."""

import numpy as np
import pytest
import torch

from test_gpu_one_call import _check_against_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 31, 32, 33, 1000, 592 * 32, 592 * 32 + 1])
def test_moments_formed_by_the_merge(T):
    """Steps around the largest batch whose moments the merge forms, every output behind the log-probs against the oracle."""
    import paper_2605_13907_b200 as ais
    rng = np.random.default_rng(T)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T)
    d, V, P, G = 128, 520, 3, 4
    cuts = np.sort(rng.integers(0, T + 1, P * G - 1))
    offs = np.concatenate([[0], cuts, [T]]).astype(np.int32)
    H = torch.randn(T, d, generator=gen, device="cuda").to(torch.bfloat16)
    W = (torch.randn(V, d, generator=gen, device="cuda") * (1.28 / d ** 0.5)).to(torch.bfloat16)
    z = H.float() @ W.float().t()
    tokens = (z - torch.empty_like(z).exponential_(generator=gen).log_()).argmax(dim=1).to(torch.int32)
    mask = (rng.random(T) < 0.7).astype(np.uint8)
    mask[T // 2] = 3                                         # any non-zero byte counts as valid
    rewards = np.tile(np.array([1, 0, 0, 1], np.float32), P)
    rewards[G:2 * G] = 1.0                                   # a prompt without a learning signal
    s = ais.AisStep(T, d, V, P, G, 128)
    s.workspace.fill_(0xA5)
    s.step(H, W, tokens, torch.from_numpy(mask).cuda(), torch.from_numpy(offs).cuda(), torch.from_numpy(rewards).cuda())
    torch.cuda.synchronize()
    assert int(s.status.item()) == 0
    _check_against_oracle(s, dict(mask=(mask != 0).astype(np.uint8), seq_offsets=offs, rewards=rewards), P, G, T)
