"""ais_step runs "each stage exactly as its own entry point does": also when a later stage is refused."""

import ctypes

import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

ERR_WORKSPACE = -4
GUARD = 4096


class Call:
    """A small step's tensors and the argument struct over them, for calls with single arguments changed."""

    def __init__(self, block=128, workspace_bytes=None):
        import paper_2605_13907_b200 as ais
        from paper_2605_13907_b200 import binding
        self.ais, self.binding = ais, binding
        w = workloads.scaled(workloads.WORKLOADS["tiny"], d=256, V=1032, P=2, G=3, lengths="uniform:40:90", block=block, seed=71)
        b = workloads.make_batch(w, device="cpu")
        rewards = torch.zeros(w.P * w.G)
        rewards[::2] = 1.0
        self.inputs = dict(H=b.H.cuda(), W=b.W.cuda(), tokens=b.tokens.cuda(), mask=b.mask.cuda(), seq_offsets=b.seq_offsets.cuda(),
                           rewards=rewards.cuda())
        self.step = s = ais.AisStep(b.T, w.d, w.V, w.P, w.G, block)
        self.out = dict(qH=s.qH, sH=s.sH, qW=s.qW, sW=s.sW, lp_train=s.lp_train, lse_train=s.lse_train, lp_roll=s.lp_roll, lse_roll=s.lse_roll,
                        adv=s.adv, n_valid_seq=s.n_valid_seq, rho=s.rho, w_tilde=s.w_tilde, diag=s.diag, dH=s.dH, loss=s.loss)
        for t in self.out.values():
            t.fill_(7)
        self.out["dev_status"] = s.status

    def run(self, stages, **changed):
        s = self.step
        args = {k: t.data_ptr() for k, t in {**self.inputs, **self.out}.items()}
        args.update(ldsH=s.sH.stride(0) if s.sH.dim() == 2 else 0, ldsW=s.sW.stride(0) if s.sW.dim() == 2 else 0,
                    workspace=s.workspace.data_ptr(), workspace_bytes=s.workspace.numel())
        args.update(changed)
        a = self.binding.StepArgs(**args)
        st = self.ais.lib().ais_step(ctypes.byref(s.shape), ctypes.byref(s.params), ctypes.byref(a), stages, None)
        torch.cuda.synchronize()
        return st

    def least_workspace_of_logprob_fwd(self):
        """Smallest size that ais_logprob_fwd accepts (with no pass asked for it enqueues nothing)."""
        s, i = self.step, self.inputs
        lo, hi = 0, s.workspace.numel()
        while lo + 1 < hi:
            mid = (lo + hi) // 2
            st = self.ais.lib().ais_logprob_fwd(ctypes.byref(s.shape), ctypes.byref(s.params), None, None, None, None, 0, None, None, 0,
                                                i["tokens"].data_ptr(), i["mask"].data_ptr(), None, None, None, None, None,
                                                s.workspace.data_ptr(), mid, None)
            assert st in (0, ERR_WORKSPACE)
            lo, hi = (lo, mid) if st == 0 else (mid, hi)
        return hi


def _stages(*names):
    from paper_2605_13907_b200 import binding
    return sum(getattr(binding, "STAGE_" + n) for n in names)


def test_a_workspace_for_the_log_probs_alone_is_not_written_behind():
    """Room for the log-probs and not for the diagnostics: the first are formed, the second refused, and nothing is touched
    behind the workspace or of what the diagnostics write."""
    c = Call()
    n = c.least_workspace_of_logprob_fwd()
    ref = Call()
    assert ref.run(_stages("QUANTIZE_H", "QUANTIZE_W", "LOGPROB")) == 0
    ws = torch.full((n + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
    assert c.run(_stages("QUANTIZE_H", "QUANTIZE_W", "LOGPROB", "DIAGNOSE"), workspace=ws.data_ptr(), workspace_bytes=n) == ERR_WORKSPACE
    assert bool((ws[n:] == 0xA5).all())
    for name in ("adv", "n_valid_seq", "rho", "w_tilde", "diag"):
        assert bool((c.out[name] == 7).all()), name
    for name in ("lp_train", "lse_train", "lp_roll", "lse_roll"):
        assert torch.equal(c.out[name], ref.out[name]), name


@pytest.mark.parametrize("refused", ["dH", "lse_train", "workspace", "lddw"])
def test_a_refused_loss_leaves_the_stages_before_it_whole(refused):
    """The diagnostics of a call whose loss stage is refused: the same bits as without that stage."""
    before = _stages("QUANTIZE_H", "QUANTIZE_W", "LOGPROB", "DIAGNOSE")
    c, ref = Call(), Call()
    assert ref.run(before) == 0
    dW = torch.empty(1032, 256, device="cuda")
    changed = {"dH": dict(dH=None), "lse_train": dict(lse_train=None), "lddw": dict(dW=dW.data_ptr(), lddw=128),
               "workspace": dict(workspace_bytes=c.ais.workspace_min_bytes(c.step.shape, c.step.params) - 1)}[refused]
    assert c.run(before | _stages("LOSS"), **changed) < 0
    for name in ("lp_train", "lp_roll", "adv", "n_valid_seq", "rho", "w_tilde", "diag"):
        assert torch.equal(c.out[name], ref.out[name]), name
    assert bool((c.out["dH"] == 7).all()) and float(c.out["loss"]) == 7.0


@pytest.mark.parametrize("block", [128, 0])
@pytest.mark.parametrize("why", ["no pass asked for", "log-probs refused", "codes of W refused"])
def test_codes_are_written_whatever_becomes_of_the_log_probs(why, block):
    """Quantisers that ais_step merges into the log-probs' opening launch run without it, too."""
    c, ref = Call(block), Call(block)
    assert ref.run(_stages("QUANTIZE_H", "QUANTIZE_W")) == 0
    changed = {"no pass asked for": dict(lp_train=None, lp_roll=None), "log-probs refused": dict(tokens=None),
               "codes of W refused": dict(qW=None)}[why]
    st = c.run(_stages("QUANTIZE_H", "QUANTIZE_W", "LOGPROB"), **changed)
    assert (st == 0) == (why == "no pass asked for")
    for name in ("qH", "sH") + (("qW", "sW") if why != "codes of W refused" else ()):
        assert torch.equal(c.out[name], ref.out[name]), name
    for name in ("lp_train", "lp_roll"):
        assert bool((c.out[name] == 7).all()), name
