"""The bf16 spill of the draft's tiles 2^(z log2e - ref2): rows whose logits lie far above the reference, on both sides
of the condition for the second pass, and rows whose draft is close to its target, whose gradient is a small difference."""
import numpy as np
import pytest
import torch

import hass_inputs as hi
import oracle
from parity import compare, compare_variant

pytestmark = pytest.mark.gpu


def _hass():
    import paper_2408_15766_b200 as hass
    return hass


def _cpu(out):
    return {k: v.cpu() for k, v in out.items() if k != "workspace"}


def _second_pass(ws):
    """Word 1 of the status block: the sweep asked for the second pass."""
    return int(ws[4:8].view(torch.int32)[0]) != 0


# The sweep asks for the second pass where a lane's sum of 2^(z log2e - ref2), ref2 = z_ref log2e + 64, reaches 1e20: a
# logit (ln 1e20 + 64 ln 2) = 90.4 above the reference. Both sides with a few units to spare for the rows' noise, then
# up to and beyond the 131 at which the sum leaves the range of fp32.
@pytest.mark.parametrize("spread,redo", [(86.0, False), (95.0, True), (115.0, True), (125.0, True), (129.5, True),
                                         (131.0, True), (135.0, True)])
def test_every_spread_of_a_row_gives_the_oracle_s_gradient(spread, redo):
    """A flat target whose Top-K tokens the draft holds at -60, one token of every third row `spread` above them, weights
    of 1/8192: the row scale of the spill, g S_q e^(ref - lse_d), is the smallest number of the path."""
    hass = _hass()
    N, d, V, K = 200, 64, 3000, 4
    inp = hi.make_custom(N, d, V, K, seed=9, sigma_w=0.05)
    W = inp.W.clone()
    W[:, :2] = 0
    W[:256, 0] = 1.0                    # tokens 0 .. 255: the target's favourites, about 3 above the others, at -60 in the draft
    W[2000, 1] = 0.5
    H_t, H_d = inp.H_t.clone(), inp.H_d[0].clone()
    H_t[:, 0], H_t[:, 1] = 3.0, 0.0
    H_d[:, 0], H_d[:, 1] = -60.0, 0.0
    H_d[::3, 1] = 2.0 * (spread - 60.0)      # token 2000
    grad = np.random.default_rng(1).uniform(0.5, 1.5, size=N) / 8192
    dev = torch.device("cuda:0")
    g = torch.tensor(grad, dtype=torch.float32, device=dev)
    args = H_t.to(dev), H_d.to(dev), W.to(dev), K
    kw = dict(grad_loss=g, dH_dtype=hass.HASS_FP32)
    out = hass.topk_distill_fwd_bwd(*args, **kw)
    hass.check(out["workspace"])
    assert _second_pass(out["workspace"]) == redo
    print("fused", compare(H_t, H_d, W, K, _cpu(out), grad_loss=grad))
    s2 = hass.topk_distill_fwd_bwd_draft(args[1], args[2], out["topk_idx"], out["topk_q"], workspace=out["workspace"], **kw)
    hass.check(out["workspace"])
    assert _second_pass(out["workspace"]) == redo
    print("draft", compare(H_t, H_d, W, K, dict(_cpu(out), **_cpu(s2)), grad_loss=grad))
    v = hass.variant_distill_fwd_bwd(*args, hass.LOSS_TOP_P, 0.004, **kw)
    hass.check(v["workspace"])
    assert _second_pass(v["workspace"]) == redo
    print("top-p", compare_variant(H_t, H_d, W, K, oracle.VARIANT_TOP_P, 0.004, _cpu(v), grad_loss=grad))
    v = hass.variant_distill_fwd_bwd(*args, hass.LOSS_BIDIR_TOPK, 0.0, **kw)
    hass.check(v["workspace"])
    assert _second_pass(v["workspace"]) == redo
    print("bidir", compare_variant(H_t, H_d, W, K, oracle.VARIANT_BIDIR, 0.0, _cpu(v), grad_loss=grad))
    c = hass.combined_distill_fwd_bwd(*args, w_topk=0.5, **kw)
    hass.check(c["workspace"])
    assert _second_pass(c["workspace"]) == redo
    cpu = _cpu(c)
    print("combined", compare(H_t, H_d, W, K, cpu, check_dH=False))
    ref = oracle.objective_from_features(hi.bf16_bits(H_t), hi.bf16_bits(H_d), hi.bf16_bits(W), K, 1.0, 0.5, grad_loss=grad,
                                         forced_idx=cpu["topk_idx"].numpy().astype(np.int32))
    ce = cpu["loss_ce"].numpy()
    assert np.all(np.abs(ce - ref["loss_ce"]) <= 2e-3 * np.abs(ref["loss_ce"]))
    assert np.abs(cpu["dH_d"].numpy().astype(np.float64) - ref["dH_d"]).max() <= 1e-2 * np.abs(ref["dH_d"]).max()


# dz_d at a token of Omega_hat is S_q p - q. With p within 1 % of q, rounding p to bf16 (2^-9) before q is taken off leaves
# 2.4e-2 of the largest gradient entry or more; the difference rounded once 2e-3 (float64 simulation of both).
@pytest.mark.parametrize("redo", [False, True])
def test_gradient_of_a_draft_close_to_its_target(redo):
    """With redo one other row lies beyond the range of its spill, so that the second pass computes every row again."""
    hass = _hass()
    N, d, V, K = 200, 64, 700, 64
    inp = hi.make_custom(N, d, V, K, seed=5, sigma_w=0.5)
    H_t, W = inp.H_t.clone(), inp.W
    H_t[:, 0] = 1.0
    H_d = H_t.clone()
    H_d[:, 0] = 1.0 + 2.0 ** -7
    if redo:
        H_d[0] = -20.0 * H_t[0]
    dev = torch.device("cuda:0")
    rows = np.arange(1, N)
    out = hass.topk_distill_fwd_bwd(H_t.to(dev), H_d.to(dev), W.to(dev), K, dH_dtype=hass.HASS_FP32)
    hass.check(out["workspace"])
    assert _second_pass(out["workspace"]) == redo
    print(compare(H_t, H_d, W, K, _cpu(out), rows=rows))
    s2 = hass.topk_distill_fwd_bwd_draft(H_d.to(dev), W.to(dev), out["topk_idx"], out["topk_q"], dH_dtype=hass.HASS_FP32,
                                         workspace=out["workspace"])
    hass.check(out["workspace"])
    print(compare(H_t, H_d, W, K, dict(_cpu(out), **_cpu(s2)), rows=rows))
