"""Dot products with, and sums of, gathered rows of W: the loss variants whose tokens are known only after the sweep."""
import numpy as np
import pytest
import torch

import hass_inputs as hi
import oracle
from parity import compare_variant

pytestmark = pytest.mark.gpu


# 8 columns a thread, 256 threads a row, 8 rows of W at a time: the narrowest rows that take all threads for one token each, a second turn of
# one thread and of all but one; sets of less than, exactly and just above one and two groups of tokens (Bi-directional ones have up to 2 K)
@pytest.mark.parametrize("d", [1800, 2048, 2056, 4088])
@pytest.mark.parametrize("K", [1, 4, 5, 8, 9, 17])
def test_gathered_rows_against_the_oracle(d, K):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    N, V = 260, 2100
    inp = hi.make_custom(N, d, V, K, seed=d + K, sigma_w=0.05)
    args = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev), K
    grad = np.random.default_rng(K).uniform(-1.0, 1.0, size=N)
    kw = dict(grad_loss=torch.tensor(grad, dtype=torch.float32, device=dev), dH_dtype=hass.HASS_FP32)
    rows = np.arange(0, N, 9)
    for variant, which in ((hass.LOSS_NORMED_TOPK, oracle.VARIANT_NORMED), (hass.LOSS_BIDIR_TOPK, oracle.VARIANT_BIDIR)):
        if variant == hass.LOSS_NORMED_TOPK and K == 1:
            continue      # constant: no loss and no gradient
        out = hass.variant_distill_fwd_bwd(*args[:3], K, variant, **kw)
        hass.check(out["workspace"])
        print(which, compare_variant(inp.H_t, inp.H_d[0], inp.W, K, which, 0.0, {k: v.cpu() for k, v in out.items() if k != "workspace"},
                                     grad_loss=grad, rows=rows))
