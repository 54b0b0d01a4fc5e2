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
