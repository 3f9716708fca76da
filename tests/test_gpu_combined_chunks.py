"""Combined calls of more than two row tiles: chunks of rows whose logits go through the workspace in fp32, two blocks of the row kernel per SM."""
import numpy as np
import pytest
import torch

import hass_inputs as hi
import oracle
from parity import compare

pytestmark = pytest.mark.gpu


# The first row of the route; one chunk, and one row more (two of ten and nine tiles, one row in the last); the largest vocabulary whose chunks
# stay in the L2 (4736 rows on 148 SMs) and one chunk of it and a row; rows of a block's first step and of one logit more; all tokens; K = 256; rows of
# which a thread of the row kernel has more pieces than a warp has lanes (512 and 1024 threads)
@pytest.mark.parametrize("N,d,V,K", [(257, 64, 9000, 10), (2304, 16, 4097, 3), (2305, 16, 4097, 3), (4737, 8, 3300, 2), (300, 72, 8192, 100),
                                     (300, 64, 8193, 256), (333, 64, 200, 200), (300, 8, 66000, 5), (3, 8, 140000, 7)])
def test_combined_chunks_against_the_oracle(N, d, V, K):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=0.3)
    args = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev), K
    grad = np.random.default_rng(N).uniform(-1.0, 1.0, size=N)
    kw = dict(w_topk=0.5, grad_loss=torch.tensor(grad, dtype=torch.float32, device=dev), dH_dtype=hass.HASS_FP32)
    out = hass.combined_distill_fwd_bwd(*args, **kw)
    hass.check(out["workspace"])
    cpu = {k: v.cpu() for k, v in out.items() if k != "workspace"}
    rows = np.unique(np.concatenate([np.arange(0, N, 13), [N - 1]]))
    print("top-k part", compare(inp.H_t, inp.H_d[0], inp.W, K, cpu, check_dH=False, rows=rows))
    ref = oracle.objective_from_features(hi.bf16_bits(inp.H_t), hi.bf16_bits(inp.H_d[0]), hi.bf16_bits(inp.W), K, 1.0, 0.5, grad_loss=grad,
                                         forced_idx=cpu["topk_idx"].numpy().astype(np.int32))
    # lse_d and z_d are fp32, of sums of d products: 1e-6 of either, and the cross-entropy is a mean of their differences
    assert np.all(np.abs(cpu["loss_ce"].numpy() - ref["loss_ce"]) <= 1e-4 * np.abs(ref["loss_ce"]))
    # every entry of dz_d is rounded to bf16 once (2^-9 of it), of which the product keeps the size at most
    scale = np.abs(ref["dH_d"]).max()
    assert np.abs(cpu["dH_d"].numpy().astype(np.float64) - ref["dH_d"]).max() <= 2.0 ** -8 * scale
    if N > 1000 or N < 128:
        return
    # a workspace without that room takes the spill, whose entries are rounded once for q and once for p
    small = torch.empty(hass.combined_distill_workspace_bytes(N, d, V, K) - 256, dtype=torch.uint8, device=dev)
    other = hass.combined_distill_fwd_bwd(*args, **kw, workspace=small)
    hass.check(small)
    assert torch.equal(other["topk_idx"], out["topk_idx"])
    assert float((other["dH_d"] - out["dH_d"]).abs().max()) <= 1e-2 * scale
