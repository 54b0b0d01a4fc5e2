"""Timing cases of the LM-head step: what a training program has the library do, at the sizes it meets.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare(case, seed)`` makes what a program
holds before the call, ``run(state)`` is one pass through the package's public entry points, ``work(case)`` states the
bytes and operations that pass cannot do without and ``tolerance(case)`` how far two correct results may lie apart.

A case is one of seven operations:

  step      quantise H and W, both log-prob passes, diagnostics, loss and dH: one (micro-)batch of a GRPO update
  grad      the same with the LM head's own gradient, the PPO ratio to an older policy and the KL term
  score     log-probs only, the head's codes kept from an earlier call (scoring responses, evaluating a policy)
  compact   scattered masks: pack the valid rows, run the step on them, scatter the results back
  quantize  the head's codes and scales anew, as after every optimiser step
  diagnose  ratios, diagnostics, mixing coefficient and corrected weights from log-probs that are already there
  static    trainer log-probs without a workspace

``block`` is the FP8 scale block (128, 64, 32), 0 for one scale per tensor, -32 / -4 for microscaling FP8 / FP4.
``dv`` is the head stored [d, V].  Sequence lengths are ragged and differ from seed to seed; their sum T does not.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2605_13907_b200 as ais

WORKSPACE_CAP = 24 << 30         # backward scratch a program sets aside at most (bytes)
SAMPLE_CELLS = 1 << 28           # logits held at once while the sampled tokens are drawn


def _case(name, op, d, V, T, P, G, block=128, dv=False, valid=False):
    return dict(name=name, op=op, d=d, V=V, T=T, P=P, G=G, block=block, dv=dv, valid=valid)


def listed():
    return [
        # the smallest batch, d=256, V=1024, 2 x 4 responses of 64 tokens: launches and host work count
        _case("tiny_step", "step", 256, 1024, 512, 2, 4),
        # one response of a few hundred tokens scored under the Qwen3-8B head
        _case("score_one_response", "score", 4096, 151936, 613, 1, 1),
        # two prompts with eight short answers each (classification or multiple choice), whole step
        _case("step_short_answers", "step", 4096, 151936, 901, 2, 8),
        # a micro-batch: one group of eight responses of 256 to 2048 tokens
        _case("step_one_group", "step", 4096, 151936, 9217, 1, 8),
        # the benchmark's batch: 8 x 8 responses, one of the eight prompts without a learning signal
        _case("step_qwen3_8b", "step", 4096, 151936, 70811, 8, 8),
        # the large-vocabulary shape with scale blocks of 32
        _case("step_large_vocab", "step", 5120, 262144, 10003, 1, 4, block=32),
        # masked diffusion: 32 responses of 512 positions, a random share of each valid, packed before the step
        _case("compact_llada_8b", "compact", 4096, 126464, 16384, 4, 8, valid=True),
        # head stored [d, V], trained itself: dH and dW, PPO ratio and KL term
        _case("grad_head_dv", "grad", 4096, 151936, 9217, 1, 8, dv=True),
        # microscaling FP8 rollouts: a group's log-probs under both policies
        _case("score_mxfp8", "score", 4096, 151936, 9217, 1, 8, block=-32),
        # the head's codes after an optimiser step
        _case("quantize_head", "quantize", 4096, 151936, 151936, 1, 1),
        # diagnostics of a long chain-of-thought batch, 32 x 16 responses
        _case("diagnose_long_cot", "diagnose", 4096, 151936, 1476661, 32, 16),
        # trainer log-probs of a 1,024-token slice where no workspace can be had
        _case("static_slice", "static", 4096, 151936, 1024, 1, 1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(["step", "step", "step", "grad", "score", "score", "compact", "quantize", "diagnose", "static"])
    small = op in ("step", "score") and rng.random() < 0.2            # test-sized heads, down to the tiny batch
    block = rng.choice([128, 128, 128, 64, 32, 0, -32, -4]) if op in ("step", "score", "quantize") else 128
    dv = op in ("step", "grad", "quantize") and block > 0 and rng.random() < 0.25
    unit = 256 if block == -4 else 128
    d = unit * (rng.randint(256 // unit, 1024 // unit) if small else rng.randint(2048 // unit, 5120 // unit))
    V = 8 * int(_log(rng, 1024, 16384) / 8) if small else 8 * int(_log(rng, 32000, 262144) / 8)
    P, G = rng.randint(1, 8), rng.choice([2, 4, 8, 8, 16])
    most = 70811.0 * 4096 * 151936 / (d * V) / (2 if op == "grad" else 1)         # rows at the largest listed case's cost
    if op == "quantize":
        P = G = 1
        T = V
    elif op == "diagnose":
        P, G = rng.randint(1, 32), rng.choice([4, 8, 16])
        T = int(_log(rng, 4096, 1476661))
    elif op == "static":
        P = G = 1
        T = int(_log(rng, 64, 16384))
    elif op == "score":
        G = rng.choice([1, 1, 4, 8])
        T = int(_log(rng, max(64, P * G), min(8192 if small else 32768, most)))
    elif op == "compact":
        T = 512 * P * G
        while T > min(65536, most) and G > 1:
            G //= 2
            T = 512 * P * G
    else:
        T = int(_log(rng, max(256, 8 * P * G), max(1024, min(8192 if small else 65536, most))))
    c = _case("", op, d, V, T, P, G, block=block, dv=dv, valid=op == "compact")
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------ inputs
def _lengths(case, rng):
    """Ragged lengths with sum T: uniform over a factor of eight, like responses of 256 to 2048 tokens."""
    S, T = case["P"] * case["G"], case["T"]
    if case["op"] == "compact":
        return np.full(S, T // S, dtype=np.int64)
    w = rng.uniform(1.0, 8.0, S)
    n = np.maximum(1, np.floor(w / w.sum() * T).astype(np.int64))
    n[int(np.argmax(n))] += T - int(n.sum())
    return n


def _live_prompts(P):
    return sum(1 for p in range(P) if p % 8 != 7)


def _rewards(case, rng):
    """0 / 1 rewards; every eighth prompt has none right and so gives no gradient, the others have some right."""
    P, G = case["P"], case["G"]
    r = np.zeros((P, G), dtype=np.float32)
    for p in range(P):
        if p % 8 != 7 and G > 1:
            r[p, rng.choice(G, size=1 + p % (G - 1), replace=False)] = 1.0
    return r.reshape(-1)


def _valid_counts(case):
    """Valid rows per sequence of a masked-diffusion batch: the mask ratios of the sequences spread evenly over (0, 1]."""
    S = case["P"] * case["G"]
    L = case["T"] // S
    return [max(1, math.ceil(L * (s + 1) / S)) for s in range(S)]


def _valid_rows(case):
    return sum(_valid_counts(case)) if case["valid"] else case["T"]


def _hidden(T, d, gen):
    """Hidden states after an RMS norm, bf16."""
    H = torch.empty(T, d, dtype=torch.bfloat16, device="cuda")
    rows = max(1, (1 << 26) // d)
    for r0 in range(0, T, rows):
        h = torch.randn(min(rows, T - r0), d, generator=gen, device="cuda")
        H[r0:r0 + rows] = h * torch.rsqrt(h.pow(2).mean(dim=1, keepdim=True) + 1e-6)
    return H


def _head(V, d, gen):
    """LM head, one row per vocabulary entry; logits of unit order at every width."""
    W = torch.empty(V, d, dtype=torch.bfloat16, device="cuda")
    rows = max(1, (1 << 26) // d)
    for r0 in range(0, V, rows):
        W[r0:r0 + rows] = torch.randn(min(rows, V - r0), d, generator=gen, device="cuda") * (1.28 / math.sqrt(d))
    return W


def _sample(H, W, gen):
    """Tokens drawn from the softmax of the logits (largest logit minus log of an exponential variate)."""
    T, V = H.shape[0], W.shape[0]
    out = torch.empty(T, dtype=torch.int32, device="cuda")
    rows = max(1, SAMPLE_CELLS // V)
    for r0 in range(0, T, rows):
        z = (H[r0:r0 + rows] @ W.t()).float()
        e = torch.empty_like(z).exponential_(generator=gen).clamp_(min=1e-20)
        out[r0:r0 + rows] = z.sub_(e.log_()).argmax(dim=1).to(torch.int32)
    return out


class _State:
    pass


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    d, V, T, P, G, block, op = (case[k] for k in ("d", "V", "T", "P", "G", "block", "op"))
    dv = case["dv"]
    s = _State()
    s.op, s.block, s.dv = op, block, dv
    f32 = dict(dtype=torch.float32, device="cuda")

    if op == "quantize":
        s.W = _head(V, d, gen)
        if dv:
            s.W = s.W.t().contiguous()
            s.codes, s.scales = ais.quantize_fp8_cols(s.W, block)
        else:
            s.codes, s.scales = ais.quantize_fp8(s.W, block)
        # a matrix of other values between this one's passes: nothing of the result is there beforehand
        s.codes.zero_()
        s.scales.zero_()
        return s

    lengths = _lengths(case, rng)
    offsets = np.zeros(P * G + 1, dtype=np.int64)
    np.cumsum(lengths, out=offsets[1:])
    s.offsets = torch.from_numpy(offsets.astype(np.int32)).cuda()
    s.rewards = torch.from_numpy(_rewards(case, rng)).cuda()

    if op == "diagnose":
        # surprisals of a sampled chain of thought (most tokens nearly certain) and the gap FP8 rollouts show
        s.lp_train = -torch.empty(T, **f32).exponential_(generator=gen).pow_(2).mul_(0.25)
        s.lp_roll = (s.lp_train + 0.03 * torch.randn(T, generator=gen, device="cuda")).clamp_(max=0.0)
        s.mask = torch.ones(T, dtype=torch.uint8, device="cuda")
        s.shape, s.params = ais.make_shape(T, d, V, P, G, block), ais.default_params()
        s.workspace = torch.empty(ais.workspace_min_bytes(s.shape, s.params), dtype=torch.uint8, device="cuda")
        s.adv, s.rho, s.w_tilde = torch.empty(P * G, **f32), torch.empty(T, **f32), torch.empty(T, **f32)
        s.n_valid_seq = torch.empty(P * G, dtype=torch.int32, device="cuda")
        s.diag = torch.zeros(19, dtype=torch.float64, device="cuda")
        return s

    s.H = _hidden(T, d, gen)
    W = _head(V, d, gen)
    s.tokens = _sample(s.H, W, gen)
    s.W = W.t().contiguous() if dv else W
    mask = np.ones(T, dtype=np.uint8)
    if case["valid"]:
        mask[:] = 0
        for i, k in zip(rng.permutation(P * G), _valid_counts(case)):
            mask[offsets[i] + rng.choice(lengths[i], size=k, replace=False)] = 1
    s.mask = torch.from_numpy(mask).cuda()

    if op == "static":
        s.shape = ais.make_shape(T, d, V, P, G, block)
        s.lp_train, s.lse_train = torch.empty(T, **f32), torch.empty(T, **f32)
        s.status = torch.zeros(1, dtype=torch.int32, device="cuda")
        return s

    params = ais.default_params(beta_kl=0.01) if op == "grad" else ais.default_params()
    s.n = _valid_rows(case)
    s.step = ais.AisStep(s.n, d, V, P, G, block, params=params, workspace_bytes_cap=WORKSPACE_CAP, want_grad=op != "score",
                         w_layout=ais.W_DV if dv else ais.W_VD)
    if op == "score":
        s.step.quantize_weights(s.W)
    if op == "grad":
        # log-probs under an older policy and the reference policy: near what this head gives the sampled tokens
        ais.logprob_fwd(s.step.shape, params, s.H, s.W, None, None, None, None, s.tokens, s.mask, s.step.lp_train,
                        s.step.lse_train, None, None, s.step.status, s.step.workspace)
        s.lp_old = s.step.lp_train + 0.05 * torch.randn(T, generator=gen, device="cuda")
        s.lp_ref = s.step.lp_train + 0.1 * torch.randn(T, generator=gen, device="cuda")
        s.dW = torch.empty(s.W.shape, **f32)
    if op == "compact":
        s.packed_mask = torch.ones(s.n, dtype=torch.uint8, device="cuda")
        s.dH = torch.empty(T, d, dtype=torch.bfloat16, device="cuda")
    return s


# ------------------------------------------------------------------------------------------ one pass
def _results(st):
    out = dict(lp_train=st.lp_train, lse_train=st.lse_train, lp_roll=st.lp_roll, lse_roll=st.lse_roll, adv=st.adv,
               n_valid_seq=st.n_valid_seq, rho=st.rho, w_tilde=st.w_tilde, diag=st.diag, loss=st.loss, dH=st.dH,
               status=st.status)
    return out


def run(s):
    if s.op == "quantize":
        if s.dv:
            return ais.quantize_fp8_cols(s.W, s.block, s.codes, s.scales)
        return ais.quantize_fp8(s.W, s.block, s.codes, s.scales)
    if s.op == "diagnose":
        ais.diagnostics(s.shape, s.params, s.lp_train, s.lp_roll, s.mask, s.offsets, s.rewards, s.adv, s.n_valid_seq, s.rho,
                        s.w_tilde, s.diag, s.workspace)
        return s.adv, s.n_valid_seq, s.rho, s.w_tilde, s.diag
    if s.op == "static":
        ais.logprob_train_static(s.shape, s.H, s.W, s.tokens, s.mask, s.lp_train, s.lse_train, s.status)
        return s.lp_train, s.lse_train, s.status
    st = s.step
    if s.op == "score":
        st.forward(s.H, s.W, s.tokens, s.mask, requantize_w=False)
        return st.lp_train, st.lse_train, st.lp_roll, st.lse_roll, st.status
    if s.op == "grad":
        st.forward(s.H, s.W, s.tokens, s.mask)
        st.diagnose(s.mask, s.offsets, s.rewards)
        st.backward(s.H, s.W, s.tokens, s.mask, s.offsets, lp_old=s.lp_old, lp_ref=s.lp_ref, dW=s.dW)
        return dict(_results(st), dW=s.dW)
    if s.op == "compact":
        rc = ais.RowCompaction(s.mask, s.offsets, n_packed=s.n)
        st.step(rc.gather_rows(s.H), s.W, rc.gather(s.tokens), s.packed_mask, rc.packed_offsets, s.rewards)
        return dict(_results(st), dH=rc.scatter_rows(st.dH, s.dH), lp_train=rc.scatter(st.lp_train), rho=rc.scatter(st.rho, 1.0),
                    w_tilde=rc.scatter(st.w_tilde, 1.0), row_index=rc.row_index[:s.n], packed_offsets=rc.packed_offsets)
    st.step(s.H, s.W, s.tokens, s.mask, s.offsets, s.rewards)
    return _results(st)


# ------------------------------------------------------------------------------------------ what a pass cannot do without
def work(case):
    d, V, T, block, op = (case[k] for k in ("d", "V", "T", "block", "op"))
    S = case["P"] * case["G"]
    code = d / 2 if block == -4 else d                                        # bytes of one row of codes
    scale = 4.0 / d if block == 0 else d / 32.0 if block < 0 else 4.0 * d / block
    if op == "quantize":
        return dict(bytes=V * (2.0 * d + code + scale), flops=2.0 * V * d)
    if op == "diagnose":
        return dict(bytes=T * (9.0 + 8.0) + 16.0 * S, flops=10.0 * T)
    n = _valid_rows(case)
    head, hidden = 2.0 * V * d, 2.0 * n * d
    rows = 4.0 * 8 * n
    if op == "static":
        return dict(bytes=head + hidden + 13.0 * T, flops=2.0 * n * d * V)
    if op == "score":
        return dict(bytes=head + V * (code + scale) + hidden + rows, flops=4.0 * n * d * V)
    # trainer logits, rollout logits, dH of the rows with a gradient (and dW): the recomputed softmax is not counted
    live = _live_prompts(case["P"]) / case["P"]
    flops = (4.0 + 2.0 * live + (2.0 * live if op == "grad" else 0.0)) * n * d * V
    total = head + 2.0 * hidden + rows
    if op == "grad":
        total += 4.0 * V * d
    if op == "compact":
        total += 2.0 * (T - n) * d + 12.0 * T                                 # dH rows and vectors of the masked positions
    return dict(bytes=total, flops=flops)


def tolerance(case):
    if case["op"] == "quantize":
        return "exact"                                                        # codes and scales are defined bit for bit
    if case["op"] in ("score", "static", "diagnose"):
        return {"rel": 1e-5}                                                  # fp32 sums in another order
    return {"rel": 1e-2}                                                      # dH is bf16, from bf16 probabilities
