"""Calls of at most 128 rows: the logits of both feature sets in fp32, one block per row for statistics, Top-K and dz_d."""
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


# fewer logits than threads, a thread's first piece and one logit more, a step of the pass and one logit more, all K tokens
@pytest.mark.parametrize("N,d,V,K", [(1, 64, 1024, 256), (3, 64, 300, 256), (5, 8, 9, 5), (7, 16, 4097, 128),
                                     (64, 64, 16384, 17), (65, 72, 16385, 100), (128, 64, 33000, 1), (33, 72, 1024, 64), (20, 64, 1024, 65)])
def test_rows_against_the_oracle(N, d, V, K):
    hass = _hass()
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=0.3)
    H_t, H_d, W = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev)
    g = np.random.default_rng(N).uniform(-1.0, 1.0, size=N)
    gd = torch.tensor(g, dtype=torch.float32, device=dev)
    out = hass.topk_distill_fwd_bwd(H_t, H_d, W, K, grad_loss=gd, dH_dtype=hass.HASS_FP32)
    hass.check(out["workspace"])
    print("fused", compare(inp.H_t, inp.H_d[0], inp.W, K, _cpu(out), grad_loss=g))
    draft = hass.topk_distill_fwd_bwd_draft(H_d, W, out["topk_idx"], out["topk_q"], grad_loss=gd, dH_dtype=hass.HASS_FP32)
    hass.check(draft["workspace"])
    for k in ("loss", "lse_d", "dH_d"):
        assert torch.equal(draft[k], out[k]), k
    fwd = hass.topk_distill_fwd(H_t, H_d, W, K)
    hass.check(fwd["workspace"])
    for k in ("loss", "lse_t", "lse_d", "topk_idx", "topk_q"):
        assert torch.equal(fwd[k], out[k]), k


@pytest.mark.parametrize("V,K,first", [(700, 40, 0), (5000, 1, 3000), (5000, 200, 1), (40000, 256, 17)])
def test_equal_logits_give_the_lowest_tokens(V, K, first):
    """From token `first` on all rows of W are the same, the others' logits lie below: more equal logits than the pool holds."""
    hass = _hass()
    dev = torch.device("cuda:0")
    d = 64
    H = torch.ones(3, d, dtype=torch.bfloat16, device=dev)
    W = torch.full((V, d), 0.125, dtype=torch.bfloat16, device=dev)
    W[:first] = -0.125
    out = hass.topk_distill_fwd_bwd(H, H, W, K)
    hass.check(out["workspace"])
    assert torch.equal(out["topk_idx"].cpu().long(), torch.arange(first, first + K).expand(3, K))


@pytest.mark.parametrize("N,d,V,K", [(1, 264, 8200, 20), (64, 512, 4100, 7), (100, 264, 8200, 128), (128, 8, 270000, 3)])
def test_variants_of_few_rows_against_the_oracle(N, d, V, K):
    """The Bi-directional variant takes this route for heads of 128 KB and more; its Omega_hat term stays in fp32."""
    hass = _hass()
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=0.1)
    args = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev), K
    for variant, which, param in ((hass.LOSS_BIDIR_TOPK, oracle.VARIANT_BIDIR, 0.0), (hass.LOSS_NORMED_TOPK, oracle.VARIANT_NORMED, 0.0),
                                  (hass.LOSS_TOP_P, oracle.VARIANT_TOP_P, 0.002)):
        if which == oracle.VARIANT_NORMED and K == 1:
            continue
        out = hass.variant_distill_fwd_bwd(*args, variant, param, dH_dtype=hass.HASS_FP32)
        hass.check(out["workspace"])
        print(which, compare_variant(inp.H_t, inp.H_d[0], inp.W, K, which, param, _cpu(out)))
