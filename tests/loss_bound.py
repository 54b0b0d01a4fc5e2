"""The loss against the float64 oracle evaluated on the device's own vectors, held to the size of its terms and not to its own:
the advantages of a prompt sum to zero, so the loss is a sum that cancels to a thousandth of its terms or less."""

import numpy as np

from oracle import ais as oais


def reference(lp_theta, mask, offs, adv, w_tilde, P, G, clip_eps=0.2, lp_old=None, lp_ref=None, beta_kl=0.0):
    """(loss, sum of the absolute values of its terms)."""
    lt = np.asarray(lp_theta, np.float64)
    old = lt if lp_old is None else np.asarray(lp_old, np.float64)
    adv = np.asarray(adv, np.float64)
    loss, _ = oais.loss_and_coeff(lt, old, mask, offs, adv, w_tilde, P, G, clip_eps, lp_ref=lp_ref, beta_kl=beta_kl)
    sid = oais.seq_ids(offs, len(lt))
    norm = 1.0 / (P * G * np.maximum(oais.valid_counts(mask, offs)[sid], 1))
    _, sur, _ = oais.surrogate_terms(lt, old, adv[sid], clip_eps)
    terms = np.abs(np.asarray(w_tilde, np.float64) * sur) * norm
    if lp_ref is not None and beta_kl != 0.0:
        log_r = np.asarray(lp_ref, np.float64) - lt
        terms = terms + beta_kl * np.abs(np.exp(log_r) - log_r - 1.0) * norm
    return loss, float(np.sum(np.where(np.asarray(mask).astype(bool), terms, 0.0)))


def check(loss, *args, **kw):
    """The device adds the terms in fp64 (1e-10 of their sum covers any order of a few million of them, and the last bits of
    exp) and rounds the result to fp32 once (2^-24)."""
    ref, terms = reference(*args, **kw)
    assert abs(float(loss) - ref) <= 2.0 ** -23 * abs(ref) + 1e-10 * terms, (float(loss), ref, terms)


def check_step(step, a, P, G, T, lp_old=None, lp_ref=None):
    """The same from a step's buffers; `a`: the batch as numpy arrays (mask, seq_offsets)."""
    vec = lambda t: t[:T].cpu().numpy().astype(np.float64)     # noqa: E731
    check(step.loss.item(), vec(step.lp_train), a["mask"], a["seq_offsets"], step.adv.cpu().numpy(), vec(step.w_tilde), P, G,
          clip_eps=float(step.params.clip_eps), lp_old=None if lp_old is None else vec(lp_old),
          lp_ref=None if lp_ref is None else vec(lp_ref), beta_kl=float(step.params.beta_kl))
