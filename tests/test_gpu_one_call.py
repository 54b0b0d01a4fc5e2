"""A step in one library call against the same step's stages called one by one, output by output.

The two share the quantisers, the rollout pass and the moments; the one-call form has its own trainer pass (which keeps the
exponentials), its own way to alpha, rho and w_tilde (inside the loss kernel) and its own scratch rows for dH.
"""

import numpy as np
import pytest
import torch

import loss_bound
from oracle import ais as oais

pytestmark = pytest.mark.gpu

CASES = {
    # name: (d, V, P, G, lengths, block, dv, share of valid rows, room for kept rows)
    "few_rows": (384, 1336, 2, 3, "uniform:1:60", 128, False, 1.0, None),
    "short_beside_long": (640, 2056, 3, 4, "mixed:3:2500", 64, True, 1.0, None),
    "scattered_mask": (512, 5008, 4, 4, "uniform:100:400", 32, False, 0.4, None),
    "many_rows": (256, 520, 8, 16, "uniform:256:700", 128, True, 0.95, None),
    "part_kept": (384, 2008, 2, 8, "uniform:150:400", 0, False, 1.0, 1),
    "mxfp8": (256, 1032, 1, 2, "uniform:200:900", -32, False, 1.0, None),
    "mxfp4": (512, 3000, 5, 2, "uniform:20:200", -4, False, 0.9, None),
}


def _lengths(spec, S, rng):
    kind, lo, hi = spec.split(":")
    lo, hi = int(lo), int(hi)
    n = rng.integers(lo, hi + 1, S)
    if kind == "mixed":                                     # every third sequence long, the others a handful of rows
        n = np.where(np.arange(S) % 3 == 0, rng.integers(hi // 2, hi + 1, S), rng.integers(lo, 3 * lo + 1, S))
    return n.astype(np.int64)


def _batch(name):
    d, V, P, G, spec, block, dv, share, cap = CASES[name]
    rng = np.random.default_rng(sorted(CASES).index(name) + 400)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(400)
    offs = np.concatenate([[0], np.cumsum(_lengths(spec, P * G, rng))]).astype(np.int32)
    T = int(offs[-1])
    H = torch.randn(T, d, generator=gen, device="cuda").to(torch.bfloat16)
    W = (torch.randn(V, d, generator=gen, device="cuda") * (1.28 / d ** 0.5)).to(torch.bfloat16)
    z = H.float() @ W.float().t()
    tokens = (z - torch.empty_like(z).exponential_(generator=gen).log_()).argmax(dim=1).to(torch.int32)
    mask = (rng.random(T) < share).astype(np.uint8)
    rewards = np.zeros((P, G), np.float32)
    for p in range(P):
        rewards[p, : 1 + p % (G - 1)] = 1.0
    a = dict(mask=mask, seq_offsets=offs, rewards=rewards.reshape(-1))
    return a, T, H, (W.t().contiguous() if dv else W), tokens


def _check_against_oracle(step, a, P, G, T):
    """Everything behind the log-probs against the oracle on the step's own log-probs."""
    lt, lr = (t[:T].cpu().numpy().astype(np.float64) for t in (step.lp_train, step.lp_roll))
    adv = oais.advantages(a["rewards"].astype(np.float64), G)
    assert np.max(np.abs(step.adv.cpu().numpy() - adv)) <= 2.0 ** -24
    assert np.array_equal(step.n_valid_seq.cpu().numpy(), oais.valid_counts(a["mask"], a["seq_offsets"]))
    ref = oais.diagnostics(lt, lr, a["mask"], adv[oais.seq_ids(a["seq_offsets"], T)], oais.Params())
    d = step.read_diag()
    assert d["n_valid"] == ref["n_valid"] and d["status_flags"] == 0
    # sums over fp32 weights that are good to 2^-22 each, relative to w - 1; the variances lose twice that
    for k in ("mean_w", "cv2", "ess_ratio", "alpha_ess", "d_bar", "alpha_mis", "std_A", "std_Aw", "delta_sigma", "alpha", "kl_k1",
              "mean_abs_dp"):
        assert d[k] == pytest.approx(ref[k], rel=1e-5, abs=1e-8), k
    _, rho, wbar = oais.ratios(lt, lr, a["mask"], 5.0)
    # the fast exponential: 2^-22 of its result, and the rounding of its argument times log2 e (2^-23 of the argument)
    tol = 1e-6 * (1.0 + np.abs(np.log(rho)))
    assert np.all(np.abs(step.rho[:T].cpu().numpy() / rho - 1.0) <= tol)
    w_tilde = oais.rectify(wbar, d["alpha"], a["mask"])
    assert np.all(np.abs(step.w_tilde[:T].cpu().numpy() - w_tilde) <= tol * np.maximum(wbar, 1.0))
    loss_bound.check_step(step, a, P, G, T)
    assert d["loss"] == pytest.approx(float(step.loss.item()), rel=2.0 ** -23)


@pytest.mark.parametrize("case", sorted(CASES))
def test_a_step_in_one_call_gives_what_its_stages_give(case):
    import paper_2605_13907_b200 as ais
    d, V, P, G, _, block, dv, _, cap = CASES[case]
    a, T, H, W, tokens = _batch(case)
    mask, offs, rewards = (torch.from_numpy(a[k]).cuda() for k in ("mask", "seq_offsets", "rewards"))
    steps = []
    for staged in (False, True):
        s = ais.AisStep(T, d, V, P, G, block, w_layout=ais.W_DV if dv else ais.W_VD, workspace_bytes_cap=cap)
        s.dH.fill_(7.0)
        if staged:
            s.forward(H, W, tokens, mask)
            s.diagnose(mask, offs, rewards)
            s.backward(H, W, tokens, mask, offs)
        else:
            s.step(H, W, tokens, mask, offs, rewards)
        torch.cuda.synchronize()
        assert int(s.status.item()) == 0
        _check_against_oracle(s, a, P, G, T)
        steps.append(s)
    one, two = steps
    for name in ("qH", "qW", "lp_roll", "lse_roll", "adv", "n_valid_seq"):
        assert torch.equal(getattr(one, name)[:T], getattr(two, name)[:T]), name
    # one form sums the exponentials about their maximum, the other about 0: the roundings of up to a few hundred fp32
    # additions per thread and of log and lse themselves (2^-20 each for 8 <= lse < 16) are another selection of the same
    for name in ("lp_train", "lse_train"):
        assert float((getattr(one, name) - getattr(two, name)).abs().max()) <= 2.0 ** -17, name
    # the losses of two sets of weights differ by no more than the weights do, term by term
    dw = (one.w_tilde[:T].double() - two.w_tilde[:T].double()).abs().max().item()
    _, terms = loss_bound.reference(one.lp_train[:T].cpu().numpy(), a["mask"], a["seq_offsets"], one.adv.cpu().numpy(), np.ones(T), P, G)
    assert abs(float(one.loss) - float(two.loss)) <= dw * terms + 2.0 ** -22 * abs(float(one.loss))
    # dH row by row, so that rows with a small factor count as much as the others: each form rounds its scratch to bf16 once
    # (2^-8 at most, the target column carries the row) and dH once (2^-9 as a rule)
    x, y = one.dH[:T].double(), two.dH[:T].double()
    norm = y.norm(dim=1)
    assert bool((x.norm(dim=1)[norm == 0] == 0).all())
    assert bool(((x - y).norm(dim=1) <= (2 * 2.0 ** -8 + 2 * 2.0 ** -9) * norm).all()), float(((x - y).norm(dim=1) / norm.clamp(min=1e-30)).max())
