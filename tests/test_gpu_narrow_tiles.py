"""Second GEMM of few rows and a short contraction: output tiles of 64 and 128 columns that clusters share."""
import numpy as np
import pytest
import torch

import hass_inputs as hi
from parity import compare

pytestmark = pytest.mark.gpu


# One row, rows that a cluster's CTAs do not share evenly, a whole row tile and three with one row in the last; a last tile of eight columns, of 96
# of 128, and whole ones; contractions of a few blocks and of the most, with a ragged last one
@pytest.mark.parametrize("N,d,V,K,fp32", [(1, 72, 700, 5, True), (3, 264, 2100, 10, False), (61, 520, 4001, 10, True), (64, 256, 1024, 10, False),
                                          (128, 1032, 1500, 20, True), (128, 136, 16384, 3, False), (100, 2784, 4695, 10, True), (257, 392, 1000, 10, True),
                                          (385, 1096, 2000, 64, False)])
def test_narrow_tiles_against_the_oracle(N, d, V, K, fp32):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, V, K, seed=N + d, sigma_w=1.0 / np.sqrt(d))
    grad = np.random.default_rng(N).uniform(-1.0, 1.0, size=N)
    out = hass.topk_distill_fwd_bwd(inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev), K,
                                    grad_loss=torch.tensor(grad, dtype=torch.float32, device=dev), dH_dtype=hass.HASS_FP32 if fp32 else hass.HASS_BF16)
    hass.check(out["workspace"])
    rows = np.unique(np.r_[np.arange(0, N, 5), N - 1])
    print(compare(inp.H_t, inp.H_d[0], inp.W, K, {k: v.cpu() for k, v in out.items() if k != "workspace"}, grad_loss=grad, rows=rows))
