"""The batch moments as part of the merge of the log-probs, which a step takes up to 18,944 rows (592 blocks of 32)."""

import numpy as np
import pytest
import torch

from oracle import ais as oais
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


def _many_sequences(T, P, G):
    """A batch of T rows in P x G sequences, most of them empty when they are more than the rows."""
    import paper_2605_13907_b200 as ais
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T + P)
    d, V, S = 128, 520, P * G
    rng = np.random.default_rng(T + P)
    offs = np.concatenate([[0], np.sort(rng.integers(0, T + 1, S - 1)), [T]]).astype(np.int32)
    H = torch.randn(T, d, generator=gen, device="cuda").to(torch.bfloat16)
    W = (torch.randn(V, d, generator=gen, device="cuda") * (1.28 / d ** 0.5)).to(torch.bfloat16)
    tokens = torch.randint(0, V, (T,), generator=gen, device="cuda", dtype=torch.int32)
    mask = (rng.random(T) < 0.8).astype(np.uint8)
    rewards = (rng.random(S) < 0.4).astype(np.float32)
    s = ais.AisStep(T, d, V, P, G, 128, want_grad=False)
    dev = [torch.from_numpy(x).cuda() for x in (mask, offs, rewards)]
    return s, H, W, tokens, mask, offs, rewards, dev


@pytest.mark.parametrize("T,P,G", [(1, 3, 2), (100, 8192, 8), (129, 1, 1000), (700, 43, 3)])
def test_advantages_of_the_opening_launch(T, P, G):
    """More sequences than the opening launch has threads for its row flags."""
    s, H, W, tokens, mask, offs, rewards, dev = _many_sequences(T, P, G)
    s.adv.fill_(9.0)
    s.n_valid_seq.fill_(77)
    s.step(H, W, tokens, *dev)
    torch.cuda.synchronize()
    assert np.max(np.abs(s.adv.cpu().numpy() - oais.advantages(rewards.astype(np.float64), G))) <= 2.0 ** -24
    assert np.array_equal(s.n_valid_seq.cpu().numpy(), oais.valid_counts(mask, offs))


@pytest.mark.parametrize("T,P,G", [(512, 16, 512), (1024, 8, 1024)])
def test_a_step_in_one_call_is_not_slower_than_its_stages_with_many_sequences(T, P, G):
    """The advantages are spread over as many threads in the step's opening launch as in a launch of their own: 0.4 and 0.6 of the
    stages' time with a thread per sequence, 5.6 times it with the threads that the row flags take."""
    s, H, W, tokens, _, _, _, (mask, offs, rewards) = _many_sequences(T, P, G)

    def stages():
        s.forward(H, W, tokens, mask)
        s.diagnose(mask, offs, rewards)

    def timed(call):
        times = []
        for _ in range(7):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            for _ in range(20):
                call()
            e1.record()
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        return sorted(times)[3]
    one, many = timed(lambda: s.step(H, W, tokens, mask, offs, rewards)), timed(stages)
    assert one <= 1.3 * many, (one, many)
