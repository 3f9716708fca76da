"""Sweeps of narrow features on eight epilogue warps: two threads share a row, and the second hands its statistics and list over at an item's end."""
import numpy as np
import pytest
import torch

import hass_inputs as hi
from parity import compare

pytestmark = pytest.mark.gpu


# 4096 rows: schedules of two phases, so that a CTA has a next item while the last one's words are read. 32100 tokens: the last tile has 100 columns,
# none for the second threads. K = 10: register lists on eight warps and the spill behind them; K = 64: the spill alone
@pytest.mark.parametrize("N,d,V,K", [(4096, 256, 32000, 10), (4096, 256, 32000, 64), (2795, 72, 32100, 16), (1025, 1024, 32100, 10)])
def test_repeated_calls_give_the_same_bits(N, d, V, K):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, V, K, seed=N + K, sigma_w=1.0 / np.sqrt(d))
    args = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev), K
    ws = torch.empty(hass.topk_distill_workspace_bytes(N, d, V, K), dtype=torch.uint8, device=dev)
    run = lambda: {k: v for k, v in hass.topk_distill_fwd_bwd(*args, dH_dtype=hass.HASS_FP32, workspace=ws).items() if k != "workspace"}
    first = run()
    hass.check(ws)
    for _ in range(20):
        for key, v in run().items():
            assert torch.equal(v, first[key]), key
    rows = np.unique(np.r_[0:4, 96:100, N - 100:N - 96, N - 4:N])
    print(compare(inp.H_t, inp.H_d[0], inp.W, K, {k: v.cpu() for k, v in first.items()}, rows=rows))
