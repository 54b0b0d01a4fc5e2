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


@pytest.mark.parametrize("T", [1, 33, 1000, 592 * 32, 592 * 32 + 1])
def test_diagnostics_behind_the_merge_without_a_loss(T):
    """Log-probs and diagnostics in one call: alpha, rho and w_tilde come from the rectifying kernel behind the merge, which may not
    read the log-probs ahead of it."""
    import paper_2605_13907_b200 as ais
    rng = np.random.default_rng(T + 1)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T + 1)
    d, V, P, G = 256, 1032, 2, 4
    offs = np.concatenate([[0], np.sort(rng.integers(0, T + 1, P * G - 1)), [T]]).astype(np.int32)
    H = torch.randn(T, d, generator=gen, device="cuda").to(torch.bfloat16)
    W = (torch.randn(V, d, generator=gen, device="cuda") * (1.28 / d ** 0.5)).to(torch.bfloat16)
    z = H.float() @ W.float().t()
    tokens = (z - torch.empty_like(z).exponential_(generator=gen).log_()).argmax(dim=1).to(torch.int32)
    mask = (rng.random(T) < 0.7).astype(np.uint8)
    mask[T // 2] = 1
    rewards = (rng.random(P * G) < 0.5).astype(np.float32)
    s = ais.AisStep(T, d, V, P, G, 128, want_grad=False)
    s.workspace.fill_(0xA5)
    for t in (s.lp_train, s.lp_roll, s.lse_train, s.lse_roll, s.rho, s.w_tilde, s.adv, s.diag):
        t.fill_(float("nan"))
    s.n_valid_seq.fill_(99)
    for _ in range(2):                                       # again, right behind the first
        s.step(H, W, tokens, *(torch.from_numpy(x).cuda() for x in (mask, offs, rewards)))
    torch.cuda.synchronize()
    assert int(s.status.item()) == 0
    lt, lr = (t[:T].cpu().numpy().astype(np.float64) for t in (s.lp_train, s.lp_roll))
    adv = oais.advantages(rewards.astype(np.float64), G)
    assert np.max(np.abs(s.adv.cpu().numpy() - adv)) <= 2.0 ** -24
    assert np.array_equal(s.n_valid_seq.cpu().numpy(), oais.valid_counts(mask, offs))
    ref = oais.diagnostics(lt, lr, mask, adv[oais.seq_ids(offs, T)], oais.Params())
    got = s.read_diag()
    assert got["n_valid"] == ref["n_valid"] and got["status_flags"] == 0 and got["loss"] == 0.0
    for k in ("mean_w", "cv2", "ess_ratio", "alpha_ess", "d_bar", "alpha_mis", "std_A", "std_Aw", "delta_sigma", "alpha", "kl_k1",
              "mean_abs_dp"):
        assert got[k] == pytest.approx(ref[k], rel=1e-5, abs=1e-8), k       # as _check_against_oracle
    _, rho, wbar = oais.ratios(lt, lr, mask, 5.0)
    tol = 1e-6 * (1.0 + np.abs(np.log(rho)))
    assert np.all(np.abs(s.rho[:T].cpu().numpy() / rho - 1.0) <= tol)
    assert np.all(np.abs(s.w_tilde[:T].cpu().numpy() - oais.rectify(wbar, got["alpha"], mask)) <= tol * np.maximum(wbar, 1.0))


def test_merged_moments_without_sequence_counts():
    """n_valid_seq is optional: the same bits without it, nothing written to it, and a loss that counts for itself."""
    from test_gpu_step_stages import Call, _stages
    before = _stages("QUANTIZE_H", "QUANTIZE_W", "LOGPROB", "DIAGNOSE")
    c, ref = Call(), Call()
    assert c.run(before, n_valid_seq=None) == 0 and ref.run(before) == 0
    names = ("lp_train", "lp_roll", "adv", "rho", "w_tilde")
    for name in names + ("diag",):
        assert torch.equal(c.out[name], ref.out[name]), name
    assert bool((c.out["n_valid_seq"] == 7).all())
    whole = Call()
    assert whole.run(before | _stages("LOSS"), n_valid_seq=None) == 0 and c.run(_stages("LOSS"), n_valid_seq=None) == 0
    for name in names + ("diag", "dH", "loss"):
        assert torch.equal(c.out[name], whole.out[name]), name
