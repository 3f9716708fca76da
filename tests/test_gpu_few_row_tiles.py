"""Calls of three to seven row tiles whose logits stay in fp32: the lines of the route by rows and vocabulary, on both sides."""
import numpy as np
import pytest
import torch

import hass_inputs as hi
import oracle
from parity import compare, compare_variant

pytestmark = pytest.mark.gpu


def _cpu(out):
    return {k: v.cpu() for k, v in out.items() if k != "workspace"}


# The first row; 50 us of the row kernel at 32000 tokens and one row more; 25 us, the line of calls that sweep one matrix, at 9000 and one row
# more; seven row tiles of the shortest vocabulary and one row more; one row in the last row tile and K = 256; the fewest tokens' K = 1;
# 65 us at 3072 features and one row more
@pytest.mark.parametrize("N,d,V,K", [(257, 64, 32000, 10), (408, 16, 32000, 40), (409, 16, 32000, 40), (505, 64, 9000, 5), (506, 64, 9000, 5),
                                     (896, 16, 2049, 16), (897, 16, 2049, 16), (385, 72, 4000, 256), (300, 64, 2100, 1), (531, 3072, 32000, 4), (532, 3072, 32000, 4)])
def test_few_row_tiles_against_the_oracle(N, d, V, K):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    # (0.3 sqrt(3072) = 17 would put the log-sum-exps near 70, where sums of 3072 products in fp32 are good to 3e-4, more than the comparison's 1e-4)
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=0.3 if d < 1000 else 0.05)
    H_t, H_d, W = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev)
    grad = np.random.default_rng(N).uniform(-1.0, 1.0, size=N)
    rows = np.unique(np.concatenate([np.arange(0, N, 17), [N - 1]]))
    kw = dict(grad_loss=torch.tensor(grad, dtype=torch.float32, device=dev), dH_dtype=hass.HASS_FP32)
    out = hass.topk_distill_fwd_bwd(H_t, H_d, W, K, **kw)
    hass.check(out["workspace"])
    print("fused", compare(inp.H_t, inp.H_d[0], inp.W, K, _cpu(out), grad_loss=grad, rows=rows))
    draft = hass.topk_distill_fwd_bwd_draft(H_d, W, out["topk_idx"], out["topk_q"], **kw)
    hass.check(draft["workspace"])
    print("draft", compare(inp.H_t, inp.H_d[0], inp.W, K, dict(_cpu(out), **_cpu(draft)), grad_loss=grad, rows=rows))
    fwd = hass.topk_distill_fwd(H_t, H_d, W, K)
    bwd = hass.topk_distill_bwd(H_d, W, out["topk_idx"], out["topk_q"], fwd["lse_d"], **kw)
    assert torch.equal(fwd["topk_idx"], out["topk_idx"])
    print("split", compare(inp.H_t, inp.H_d[0], inp.W, K, dict(_cpu(fwd), dH_d=bwd.cpu()), grad_loss=grad, rows=rows))
    for variant, which, param in ((hass.LOSS_TOP_P, oracle.VARIANT_TOP_P, 0.004), (hass.LOSS_NORMED_TOPK, oracle.VARIANT_NORMED, 0.0),
                                  (hass.LOSS_BIDIR_TOPK, oracle.VARIANT_BIDIR, 0.0)):
        if (which == oracle.VARIANT_BIDIR and K > 128) or (which == oracle.VARIANT_NORMED and K == 1):
            continue
        v = hass.variant_distill_fwd_bwd(H_t, H_d, W, K, variant, param, **kw)
        hass.check(v["workspace"])
        print(which, compare_variant(inp.H_t, inp.H_d[0], inp.W, K, which, param, _cpu(v), grad_loss=grad, rows=rows))
    # a workspace without room for the fp32 logits takes the spill: the same sets, the gradient within the bf16 rounding of both
    small = torch.empty(hass.topk_distill_workspace_bytes(N, d, V, K) - 256, dtype=torch.uint8, device=dev)
    other = hass.topk_distill_fwd_bwd(H_t, H_d, W, K, **kw, workspace=small)
    hass.check(small)
    assert torch.equal(other["topk_idx"], out["topk_idx"])
    assert float((other["dH_d"] - out["dH_d"]).abs().max()) <= 1e-2 * float(out["dH_d"].abs().max())
