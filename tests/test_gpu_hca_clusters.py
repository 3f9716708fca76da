"""Attention of few items, whose key tiles (forward) or elements (backward) clusters of CTAs share."""
import numpy as np
import pytest
import torch

import hass_inputs as hi
from hca_parity import rowwise_error, tilewise_error
from oracle import hca_oracle

pytestmark = pytest.mark.gpu


# On 148 SMs. Forward: pairs, fours and eights; a query tile with fewer key tiles than its cluster has CTAs (empty parts); a last tile of one
# position; draft passes that reach into the tile before the last CTA's; more passes than the last tile has positions. Backward: an element for
# every CTA and none for some (one position in the last key tile); a group of three
@pytest.mark.parametrize("B,T,H,Hkv,m", [(1, 1025, 2, 1, 3), (2, 900, 4, 4, 0), (1, 1200, 5, 1, 8), (3, 640, 6, 2, 2), (3, 124, 64, 8, 0), (2, 333, 4, 2, 3),
                                         (1, 257, 12, 4, 5), (1, 2000, 2, 2, 1), (5, 385, 3, 1, 1)])
def test_against_the_oracle(B, T, H, Hkv, m):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    inp = hi.make_hca_inputs(hi.HcaWorkload("clusters", B=B, T=T, H=H, Hkv=Hkv, m=m, seed=T))
    dO = torch.randn(inp.Q.shape, generator=torch.Generator().manual_seed(1)).to(torch.bfloat16)
    args = [x.to(dev) for x in (inp.Q, inp.K_t, inp.V_t)] + [[x.to(dev) for x in inp.K_d], [x.to(dev) for x in inp.V_d]]
    runs = []
    for _ in range(2):
        fw = hass.hca_attention_fwd(*args)
        hass.check(fw["workspace"])
        bw = hass.hca_attention_bwd(*args, fw["O"], fw["lse"], dO.to(dev))
        hass.check(bw["workspace"])
        runs.append((fw, bw))
    (fw, bw), (fw2, bw2) = runs
    assert torch.equal(fw["O"], fw2["O"]) and torch.equal(fw["lse"], fw2["lse"])
    assert torch.equal(bw["dK_t"], bw2["dK_t"]) and torch.equal(bw["dV_t"], bw2["dV_t"])
    f64 = lambda x: x.to(torch.float64).cpu().numpy()
    host = [f64(inp.Q), f64(inp.K_t), f64(inp.V_t), [f64(x) for x in inp.K_d], [f64(x) for x in inp.V_d]]
    O_ref, lse_ref = hca_oracle.hca_attention(*host)
    assert float(rowwise_error(f64(fw["O"]), O_ref).max()) <= 1e-2      # (as in the other attention tests)
    assert float(np.abs(f64(fw["lse"]) - lse_ref).max()) <= 2e-3
    ref = hca_oracle.hca_attention_grad(*host, f64(dO))
    pairs = [(bw["dQ"], ref[0]), (bw["dK_t"], ref[1]), (bw["dV_t"], ref[2])] + list(zip(bw["dK_d"], ref[3])) + list(zip(bw["dV_d"], ref[4]))
    assert max(float(tilewise_error(f64(a), b).max()) for a, b in pairs) <= 1.5e-2
