"""Calls of more than one row tile over a short vocabulary, whose logits stay in fp32, and sweeps of narrow features, whose epilogue has
eight warps."""
import numpy as np
import pytest
import torch

import hass_inputs as hi
import oracle
from parity import compare, compare_variant

pytestmark = pytest.mark.gpu


def _cpu(out):
    return {k: v.cpu() for k, v in out.items() if k != "workspace"}


# The first row of the route and the last before it; the largest calls of each row kernel (128, 256, 512 threads a row) and the first beyond;
# three row tiles of which one is shared by both matrices' pairs, one row in the last
@pytest.mark.parametrize("N,d,V,K", [(256, 64, 1024, 10), (257, 64, 1024, 32), (385, 72, 700, 3), (3072, 16, 1024, 32), (3073, 16, 1024, 32),
                                     (2048, 16, 2048, 64), (2049, 16, 1025, 33), (1024, 16, 2048, 200), (1025, 16, 1300, 65), (300, 64, 90, 90)])
def test_short_vocabularies_against_the_oracle(N, d, V, K):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=0.3)
    H_t, H_d, W = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev)
    grad = np.random.default_rng(N).uniform(-1.0, 1.0, size=N)
    kw = dict(grad_loss=torch.tensor(grad, dtype=torch.float32, device=dev), dH_dtype=hass.HASS_FP32)
    out = hass.topk_distill_fwd_bwd(H_t, H_d, W, K, **kw)
    hass.check(out["workspace"])
    print("fused", compare(inp.H_t, inp.H_d[0], inp.W, K, _cpu(out), grad_loss=grad))
    draft = hass.topk_distill_fwd_bwd_draft(H_d, W, out["topk_idx"], out["topk_q"], **kw)
    fwd = hass.topk_distill_fwd(H_t, H_d, W, K)
    bwd = hass.topk_distill_bwd(H_d, W, out["topk_idx"], out["topk_q"], fwd["lse_d"], **kw)
    hass.check(fwd["workspace"])
    assert torch.equal(fwd["topk_idx"], out["topk_idx"])
    print("split", compare(inp.H_t, inp.H_d[0], inp.W, K, dict(_cpu(fwd), dH_d=bwd.cpu()), grad_loss=grad))
    print("draft", compare(inp.H_t, inp.H_d[0], inp.W, K, dict(_cpu(out), **_cpu(draft)), grad_loss=grad))
    rows = np.arange(0, N, 7)
    c = hass.combined_distill_fwd_bwd(H_t, H_d, W, K, w_topk=0.5, **kw)
    hass.check(c["workspace"])
    ref = oracle.objective_from_features(hi.bf16_bits(inp.H_t), hi.bf16_bits(inp.H_d[0]), hi.bf16_bits(inp.W), K, 1.0, 0.5, grad_loss=grad,
                                         forced_idx=c["topk_idx"].cpu().numpy().astype(np.int32))
    assert np.all(np.abs(c["loss_ce"].cpu().numpy() - ref["loss_ce"]) <= 2e-3 * np.abs(ref["loss_ce"]))
    assert np.abs(c["dH_d"].cpu().numpy().astype(np.float64) - ref["dH_d"]).max() <= 1e-2 * np.abs(ref["dH_d"]).max()
    for variant, which in ((hass.LOSS_NORMED_TOPK, oracle.VARIANT_NORMED), (hass.LOSS_BIDIR_TOPK, oracle.VARIANT_BIDIR)):
        if which == oracle.VARIANT_BIDIR and K > 128:
            continue
        v = hass.variant_distill_fwd_bwd(H_t, H_d, W, K, variant, **kw)
        hass.check(v["workspace"])
        print(which, compare_variant(inp.H_t, inp.H_d[0], inp.W, K, which, 0.0, _cpu(v), grad_loss=grad, rows=rows))


# Lanes of three tiles and more on 148 SMs; a last tile with columns in its first half alone, of one column, and a whole one; single CTAs and
# pairs, several row tiles, the widest features of the form and the first beyond
@pytest.mark.parametrize("N,d,V,K", [(300, 72, 20000, 16), (300, 72, 19205, 1), (300, 64, 20224, 10), (2100, 1024, 6000, 16), (2100, 1032, 6000, 16),
                                     (200, 128, 38145, 40), (640, 64, 24577, 7)])
def test_narrow_features_against_the_oracle(N, d, V, K):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=0.3 if d < 1000 else 0.05)
    args = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev), K
    rows = np.unique(np.concatenate([np.arange(0, N, 31), [N - 1]]))
    out = hass.topk_distill_fwd_bwd(*args, dH_dtype=hass.HASS_FP32)
    hass.check(out["workspace"])
    print("fused", compare(inp.H_t, inp.H_d[0], inp.W, K, _cpu(out), rows=rows))
    fwd = hass.topk_distill_fwd(*args)
    hass.check(fwd["workspace"])
    print("forward", compare(inp.H_t, inp.H_d[0], inp.W, K, _cpu(fwd), rows=rows, check_dH=False))


@pytest.mark.parametrize("K", [1, 10, 16])
def test_equal_logits_of_both_halves_of_a_tile_give_the_lowest_tokens(K):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    N, d, V = 300, 64, 20000
    H = torch.ones(N, d, dtype=torch.bfloat16, device=dev)
    W = torch.zeros(V, d, dtype=torch.bfloat16, device=dev)
    W[torch.arange(V, device=dev) % 128 >= 120] = 0.125      # the last tokens of every half share the largest logit
    out = hass.topk_distill_fwd_bwd(H, H, W, K)
    hass.check(out["workspace"])
    want = torch.arange(V)[torch.arange(V) % 128 >= 120][:K]
    assert torch.equal(out["topk_idx"].cpu().long(), want.expand(N, K))
