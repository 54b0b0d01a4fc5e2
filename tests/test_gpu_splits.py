"""How the tensor-core passes split their work: vocabulary ranges of the forward and recompute passes for few row tiles, and
contraction ranges of the dH tiles that do not fill a wave.  Shapes sit at the edges of the rules (one row, one row tile,
one tile more than a wave, ranges shorter than the stage ring allows, a tail without work), against the float64 oracle.
"""

import numpy as np
import pytest
import torch

import workloads
from oracle import ais as oais

pytestmark = pytest.mark.gpu

LP_ATOL = 1e-4          # fp32 sums of d <= 2560 products of unit-order logits: d * 2^-24 * sum|h w| stays below this
DH_REL = 1e-2           # dH is bf16 (2^-9) from bf16 probabilities (2^-9)

CASES = {
    # name: (d, V, P, G, lengths)                            row tiles, dH tiles (256 x 256) and what they meet
    "one_row": (128, 256, 1, 2, "const:1"),                 # one column tile, four K steps: nothing to split
    "one_tile": (256, 5008, 1, 2, "const:64"),              # 1 row tile, 20 column tiles -> 20 ranges; 1 dH tile -> 19 ranges
    "short_ranges": (384, 1336, 2, 3, "uniform:50:130"),    # ragged columns; 21 K steps -> ranges of 4 and 5 steps
    "ragged_pairs": (640, 2056, 2, 4, "uniform:100:180"),   # half-empty last pair, ragged last column tile of dH
    "past_a_wave": (2560, 1032, 4, 8, "uniform:118:126"),   # 16 pairs x 10 = 160 tiles: a full wave and 12 split tiles
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_split_passes_match_the_oracle(case):
    import paper_2605_13907_b200 as ais
    d, V, P, G, lengths = CASES[case]
    w = workloads.scaled(workloads.WORKLOADS["tiny"], d=d, V=V, P=P, G=G, lengths=lengths, w_std=d ** -0.5, seed=301)
    b = workloads.make_batch(w, device="cpu")
    if case == "past_a_wave":
        b.mask[-600:] = 0                                   # the last row pairs have no work: their split tiles are zeros
    rewards = torch.zeros(P * G)
    rewards[::2] = 1.0                                      # every group has a learning signal
    b.rewards = rewards
    a = workloads.to_numpy(b)
    ref = oais.full_path(a["H"], a["W"], a["tokens"], a["mask"], a["seq_offsets"], a["rewards"], P, G, w.block)
    T = b.T
    step = ais.AisStep(T, d, V, P, G, w.block)
    step.dH.fill_(7.0)
    H, W, tok, msk = b.H.cuda(), b.W.cuda(), b.tokens.cuda(), b.mask.cuda()
    step.step(H, W, tok, msk, b.seq_offsets.cuda(), b.rewards.cuda())
    torch.cuda.synchronize()
    assert int(step.status.item()) == 0
    for name in ("lp_train", "lp_roll", "lse_train"):
        assert np.max(np.abs(getattr(step, name)[:T].cpu().numpy() - ref[name])) <= LP_ATOL, name
    dH = step.dH[:T].float().cpu().numpy().astype(np.float64)
    assert np.all(dH[a["mask"] == 0] == 0)
    for r in range(0, T, 256):                              # tile by tile: a range left out of one tile shows
        for c in range(0, d, 256):
            g, x = dH[r:r + 256, c:c + 256], ref["dH"][r:r + 256, c:c + 256]
            assert np.linalg.norm(g - x) <= DH_REL * max(np.linalg.norm(x), 1e-12), (r, c)
    lp = torch.empty(T, device="cuda")
    ais.logprob_train_static(step.shape, H, W, tok, msk, lp)
    assert np.max(np.abs(lp.cpu().numpy() - ref["lp_train"])) <= LP_ATOL


@pytest.mark.parametrize("dv", [False, True])
@pytest.mark.parametrize("rows", ["ordinary", "mixed"])
def test_kept_exponentials_match_the_oracle(rows, dv):
    """A step in one call keeps e^z of the forward pass for dH; rows whose log-sum-exp lies outside [-20, 59] are recomputed,
    alone or beside ordinary rows of their tile.  With room for 128 rows only the first tile is kept: same bits."""
    import paper_2605_13907_b200 as ais
    d, V, P, G = 384, 1336, 2, 3
    w = workloads.scaled(workloads.WORKLOADS["tiny"], d=d, V=V, P=P, G=G, lengths="uniform:90:130", w_std=d ** -0.5, seed=302)
    b = workloads.make_batch(w, device="cpu")
    T = b.T
    if rows == "mixed":
        b.W[:, 0] = 1.0
        b.H[:, 0] = 0.0
        b.H[0:3] *= 30.0                                    # logits beyond +-59 (first tile)
        b.H[130:150, 0] = -50.0                             # log-sum-exp near -43
        b.H[256:384:7, 0] = 70.0                            # near +77, scattered over a tile
        b.tokens[0:3] = 5                                   # a target that is far from certain
    b.mask[40:60] = 0
    rewards = torch.zeros(P * G)
    rewards[::2] = 1.0
    b.rewards = rewards
    a = workloads.to_numpy(b)
    ref = oais.full_path(a["H"], a["W"], a["tokens"], a["mask"], a["seq_offsets"], a["rewards"], P, G, w.block)
    Wx = (b.W.t().contiguous() if dv else b.W).cuda()
    out = []
    for cap in (None, 1):
        step = ais.AisStep(T, d, V, P, G, w.block, workspace_bytes_cap=cap, w_layout=ais.W_DV if dv else ais.W_VD)
        step.dH.fill_(7.0)
        step.step(b.H.cuda(), Wx, b.tokens.cuda(), b.mask.cuda(), b.seq_offsets.cuda(), b.rewards.cuda())
        torch.cuda.synchronize()
        assert int(step.status.item()) == 0
        # |z| up to 120: fp32 sums of d products and the rounding of the sum itself, 120 * 2^-23 * a few
        assert np.max(np.abs(step.lse_train[:T].cpu().numpy() - ref["lse_train"])) <= LP_ATOL
        out.append(step.dH[:T].clone())
    dH = out[0].float().cpu().numpy().astype(np.float64)
    assert np.all(dH[a["mask"] == 0] == 0)
    for r in range(0, T, 128):
        assert np.linalg.norm(dH[r:r + 128] - ref["dH"][r:r + 128]) <= DH_REL * np.linalg.norm(ref["dH"][r:r + 128]), r
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("V", [40, 64, 264, 520, 832])
def test_d_by_v_head_at_the_edges_of_the_column_blocks(V):
    """Heads stored [d, V] narrower than a 64-column block, and with whole and partial blocks and tiles at their end: the same
    log-probs bit for bit as the [V, d] form, and dH within the rounding of bf16 (2^-8) of it."""
    import paper_2605_13907_b200 as ais
    d, P, G = 256, 1, 4
    w = workloads.scaled(workloads.WORKLOADS["tiny"], d=d, V=V, P=P, G=G, lengths="uniform:30:80", w_std=d ** -0.5, seed=303)
    b = workloads.make_batch(w, device="cpu")
    out = []
    for dv in (False, True):
        step = ais.AisStep(b.T, d, V, P, G, w.block, w_layout=ais.W_DV if dv else ais.W_VD)
        W = (b.W.t().contiguous() if dv else b.W).cuda()
        step.step(b.H.cuda(), W, b.tokens.cuda(), b.mask.cuda(), b.seq_offsets.cuda(), torch.tensor([1.0, 0.0, 0.0, 1.0]).cuda())
        torch.cuda.synchronize()
        assert int(step.status.item()) == 0
        out.append(step)
    assert torch.equal(out[0].lp_train, out[1].lp_train) and torch.equal(out[0].lp_roll, out[1].lp_roll)
    a, c = out[0].dH.double(), out[1].dH.double()
    assert float((a - c).norm()) <= 2 ** -8 * float(a.norm())


@pytest.mark.parametrize("variant", ["vd", "dv", "per_tensor"])
def test_two_row_tiles_per_cta_match_the_oracle(variant):
    """Enough row tiles for 256-row units: pairs with either row tile masked, both masked, a ragged last pair with one row tile,
    rows outside the exponent form in one tile of a pair; the step in one call and the stages on their own."""
    import paper_2605_13907_b200 as ais
    d, V, P, G = 1280, 2568, 2, 4
    block = 0 if variant == "per_tensor" else 128
    dv = variant == "dv"
    w = workloads.scaled(workloads.WORKLOADS["tiny"], d=d, V=V, P=P, G=G, lengths="uniform:265:285", w_std=d ** -0.5, seed=304, block=block)
    b = workloads.make_batch(w, device="cpu")
    T = b.T
    assert T % 256 != 0
    b.mask[128:256] = 0                                     # second tile of pair 0
    b.mask[256:384] = 0                                     # first tile of pair 1
    b.mask[512:768] = 0                                     # pair 2
    b.W[:, 0] = 1.0
    b.H[:, 0] = 0.0
    b.H[900:910, 0] = 70.0                                  # second tile of pair 3: log-sum-exp near +77
    rewards = torch.zeros(P * G)
    rewards[::2] = 1.0
    b.rewards = rewards
    a = workloads.to_numpy(b)
    ref = oais.full_path(a["H"], a["W"], a["tokens"], a["mask"], a["seq_offsets"], a["rewards"], P, G, block)
    # every MMA step (16 of the d products, d / 16 of them) may cut the accumulator off at one unit of its last place: 2^-17 for
    # the logits near 77, so d / 16 * 2^-17 = 6.1e-4 there; the other rows as above
    atol = LP_ATOL + np.where(np.abs(ref["lse_train"]) > 32, d / 16 * 2.0 ** -17, 0.0)
    W = (b.W.t().contiguous() if dv else b.W).cuda()
    H, tok, msk, offs, rew = b.H.cuda(), b.tokens.cuda(), b.mask.cuda(), b.seq_offsets.cuda(), b.rewards.cuda()
    step = ais.AisStep(T, d, V, P, G, block, w_layout=ais.W_DV if dv else ais.W_VD)

    def check():
        torch.cuda.synchronize()
        assert int(step.status.item()) == 0
        for name in ("lp_train", "lp_roll", "lse_train"):
            assert np.all(np.abs(getattr(step, name)[:T].cpu().numpy() - ref[name]) <= atol), name
        dH = step.dH[:T].float().cpu().numpy().astype(np.float64)
        assert np.all(dH[a["mask"] == 0] == 0)
        for r in range(0, T, 128):
            assert np.linalg.norm(dH[r:r + 128] - ref["dH"][r:r + 128]) <= DH_REL * max(np.linalg.norm(ref["dH"][r:r + 128]), 1e-12), r

    step.dH.fill_(7.0)
    step.step(H, W, tok, msk, offs, rew)
    check()
    step.dH.fill_(7.0)
    step.backward(H, W, tok, msk, offs)
    check()
    lp = torch.empty(T, device="cuda")
    if not dv:
        ais.logprob_train_static(step.shape, H, W, tok, msk, lp)
        assert np.all(np.abs(lp.cpu().numpy() - ref["lp_train"]) <= atol)


@pytest.mark.parametrize("gaps", ["small", "mixed"])
@pytest.mark.parametrize("T", [(8 << 20) - 1, 8 << 20, (8 << 20) + 2049])
def test_long_batches_sum_their_moments_in_one_launch_or_two(T, gaps):
    """From 8 Mi rows on the exact walk over groups of tiny log-ratio gaps is a launch of its own, which replaces the sums of
    the blocks that need it: all of them ("small": every gap is 1e-4) or those of the first half ("mixed").  Tolerance: the
    weights are good to fp32 relative to w - 1 (2^-23 and the exponential's 2^-22), the sums over them are fp64."""
    import ctypes

    import paper_2605_13907_b200 as ais
    rng = np.random.default_rng(T % 1000 + len(gaps))
    P, G = 2, 4
    S = P * G
    offs = np.concatenate([[0], np.sort(rng.integers(0, T + 1, S - 1)), [T]]).astype(np.int32)
    lp_t = -rng.uniform(0.5, 4.0, T).astype(np.float32)
    size = np.full(T, 1e-4)
    if gaps == "mixed":
        size[T // 2:] = 0.3
    lp_r = (lp_t - size * rng.choice([-1.0, 1.0], T)).astype(np.float32)
    mask = (rng.random(T) < 0.8).astype(np.uint8)
    rew = np.array([1, 0, 0, 1, 0, 1, 0, 0], np.float32)
    ref_adv = oais.advantages(rew.astype(np.float64), G)
    ref = oais.diagnostics(lp_t, lp_r, mask, ref_adv[oais.seq_ids(offs, T)], oais.Params())
    params = ais.default_params()
    shape = ais.make_shape(T, 128, 1024, P, G, 128)
    ws = torch.empty(ais.workspace_min_bytes(shape, params), dtype=torch.uint8, device="cuda")
    adv, nseq = torch.empty(S, device="cuda"), torch.zeros(S, dtype=torch.int32, device="cuda")
    rho, wt = torch.zeros(T, device="cuda"), torch.zeros(T, device="cuda")
    diag = torch.zeros(32, dtype=torch.float64, device="cuda")
    ais.diagnostics(shape, params, *(torch.from_numpy(x).cuda() for x in (lp_t, lp_r, mask, offs, rew)), adv, nseq, rho, wt, diag, ws)
    d = ais.Diag.from_buffer_copy(diag.cpu().numpy().tobytes()[:ctypes.sizeof(ais.Diag)]).as_dict()
    assert d["n_valid"] == ref["n_valid"] and d["status_flags"] == 0
    assert np.array_equal(nseq.cpu().numpy(), np.add.reduceat(np.append(mask, 0).astype(np.int64), offs[:-1]) * (np.diff(offs) > 0))
    for k in ("cv2", "std_Aw", "delta_sigma", "alpha_ess", "d_bar", "kl_k1", "mean_abs_dp", "alpha"):
        assert abs(d[k] - ref[k]) <= 1e-4 * max(abs(ref[k]), 1e-9 if k == "cv2" else 1e-4), (k, d[k], ref[k])
    valid = mask.astype(bool)
    ref_wt = oais.rectify(oais.ratios(lp_t, lp_r, mask, 5.0)[2], ref["alpha"], mask)
    assert np.abs(wt.cpu().numpy() - ref_wt)[valid].max() <= 1e-5 and bool((wt.cpu()[~torch.from_numpy(valid)] == 1).all())


@pytest.mark.parametrize("dv", [False, True])
@pytest.mark.parametrize("length", [5, 17, 25, 50])
def test_weight_gradient_with_few_and_many_k_steps(length, dv):
    """dW of 40, 136, 200 and 400 rows: fewer 64-row K steps than the stage ring holds (1, 3), one more (4), and enough for the
    whole order of row tiles (7); 237 units of 256 x 256, so that CTAs have a second one; a last unit with one row tile and a
    ragged column tile.  dW is fp32 from bf16 gradients (2^-9)."""
    import paper_2605_13907_b200 as ais
    d, V, P, G = 640, 20104, 2, 4
    w = workloads.scaled(workloads.WORKLOADS["tiny"], d=d, V=V, P=P, G=G, lengths=f"const:{length}", w_std=d ** -0.5, seed=305)
    b = workloads.make_batch(w, device="cpu")
    a = workloads.to_numpy(b)
    ref = oais.full_path(a["H"], a["W"], a["tokens"], a["mask"], a["seq_offsets"], a["rewards"], P, G, w.block)
    W = (b.W.t().contiguous() if dv else b.W).cuda()
    H, tok, msk, offs, rew = b.H.cuda(), b.tokens.cuda(), b.mask.cuda(), b.seq_offsets.cuda(), b.rewards.cuda()
    step = ais.AisStep(b.T, d, V, P, G, w.block, w_layout=ais.W_DV if dv else ais.W_VD)
    dW = torch.full((d, V) if dv else (V, d), 7.0, device="cuda")
    step.forward(H, W, tok, msk)
    step.diagnose(msk, offs, rew)
    for accumulate in (False, True):
        step.backward(H, W, tok, msk, offs, dW=dW, dw_accumulate=accumulate)
        torch.cuda.synchronize()
        assert int(step.status.item()) == 0
        got = (dW.t() if dv else dW).double().cpu().numpy() / (2.0 if accumulate else 1.0)
        for c in range(0, V, 256):
            assert np.linalg.norm(got[c:c + 256] - ref["dW"][c:c + 256]) <= DH_REL * np.linalg.norm(ref["dW"][c:c + 256]), c
