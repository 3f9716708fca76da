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


# Normed Top-K shares a row's columns among two, four and eight blocks: of 257, 514 and 1027 units of eight columns the parts differ by one, and
# where the widest has 129 its threads form one group, those of a part of 128 two. (Logits of deviation 1.8: the tensor cores add d / 16 partial
# sums in fp32 without rounding to nearest, at most 2^-23 |z| each, 6e-5 |z| for d = 8216 and 7.5e-6 |z| as seen; the 1e-4 that lse_t is held to
# is below the latter where logits reach 15, as with sigma_w = 0.05, and above it up to 13.)
@pytest.mark.parametrize("N,d", [(200, 2056), (80, 4112), (30, 8216)])
@pytest.mark.parametrize("K", [8, 10])
def test_normed_rows_of_unequal_parts_against_the_oracle(N, d, K):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, 1100, K, seed=d + K, sigma_w=0.02)
    out = hass.variant_distill_fwd_bwd(inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev), K, hass.LOSS_NORMED_TOPK, dH_dtype=hass.HASS_FP32)
    hass.check(out["workspace"])
    print(compare_variant(inp.H_t, inp.H_d[0], inp.W, K, oracle.VARIANT_NORMED, 0.0, {k: v.cpu() for k, v in out.items() if k != "workspace"},
                          rows=np.arange(0, N, 7)))
