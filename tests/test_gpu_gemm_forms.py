"""The forms of the GEMM and selection kernels at the sizes where they can go wrong: CTA pairs whose last row tile has no
partner, output tiles cut along the contraction (alone, behind whole rounds, with few rows), selections of one and of
four warps per row, against the oracle with the tolerances of the parity tests, every buffer between guard bands."""
import numpy as np
import pytest
import torch

import hass_inputs as hi
from parity import compare, least_workspace
from test_gpu_parity import _guarded_fused

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d,V,K,fp32", [
    (1600, 64, 5000, 10, True),        # 13 row tiles as seven pairs, the last one with a tile of its own only
    (1537, 200, 3000, 20, False),      # the same with one row in the last tile and a ragged last column tile
    (61, 520, 20000, 10, False),       # one row tile: cut output tiles that keep 61 rows
    (129, 264, 30001, 5, True),        # two row tiles, one row in the second, a ragged contraction
    (700, 64, 9000, 200, True),        # selection of a large K with one warp per row, which cuts its pool
    (40, 64, 33000, 40, True),         # the same with four warps per row and buffers of 129 lanes
    (129, 64, 9000, 64, True),         # 127 padding rows in the second row tile, buffered candidates
    (64, 72, 33001, 256, False),       # the most rows whose draft logits go through the workspace in fp32, the largest K
    (65, 72, 33001, 256, False),       # one row more
    (128, 264, 20001, 12, True),       # the most rows of one tile; output tiles shared by clusters
    (250, 520, 20000, 10, False),      # two row tiles, output tiles shared by clusters
    (620, 64, 40000, 16, True),        # one warp per row, K lists whose first entries set the floor
    (1601, 2824, 12000, 10, False),    # whole rounds of output tiles, then a cut rest, d not a multiple of 256
])
def test_pairs_and_cut_tiles(N, d, V, K, fp32):
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=2.0 / np.sqrt(d))
    grad = np.random.default_rng(1).normal(size=N)
    rows = None if N * d * V < 3e9 else np.unique(np.r_[0:8, 120:136, N - 70:N - 60, N - 8:N])
    fused, split = _guarded_fused(inp, K, grad, dH_fp32=fp32)
    print("fused", compare(inp.H_t, inp.H_d[0], inp.W, K, fused, grad_loss=grad, rows=rows))
    print("split", compare(inp.H_t, inp.H_d[0], inp.W, K, split, grad_loss=grad, rows=rows))


@pytest.mark.parametrize("value", [3.0, 200.0])
def test_reference_exponent_far_below_the_row(value):
    """The target's first token has a low draft logit (-60): draft rows whose largest logit is 60 above it stay within the
    spill's range, rows 260 above it are redone by the second pass; both match the oracle."""
    N, d, V, K = 200, 64, 3000, 4
    inp = hi.make_custom(N, d, V, K, seed=9, sigma_w=0.05)
    W = inp.W.clone()
    W[:, 0] = 0
    W[5, 0] = 1.0                       # token 5: the target's favourite, and far down in the draft
    W[2000, 1] = 0.5
    H_t, H_d = inp.H_t.clone(), inp.H_d[0].clone()
    H_t[:, 0] = 20.0
    H_d[:, 0] = -60.0
    H_d[::3, 1] = 2.0 * value           # token 2000 at +value on every third row
    case = hi.Inputs(**{**inp.__dict__, "H_t": H_t, "H_d": [H_d], "W": W})
    fused, split = _guarded_fused(case, K, None)
    print("fused", compare(H_t, H_d, W, K, fused))
    print("split", compare(H_t, H_d, W, K, split))


@pytest.mark.parametrize("N", [60, 100, 128])
def test_one_row_tile_with_less_workspace_and_from_host_buffers(N):
    """Calls of one row tile keep their logits in fp32 where the workspace has room: with the least
    workspace the results are the oracle's too, and the entry for host buffers gives the device entry's bits."""
    import paper_2408_15766_b200 as hass
    d, V, K = 136, 5000, 10
    inp = hi.make_custom(N, d, V, K, seed=N, sigma_w=0.2)
    dev = torch.device("cuda:0")
    H_t, H_d, W = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev)
    a = hass.topk_distill_fwd_bwd(H_t, H_d, W, K)
    b = hass.topk_distill_fwd_bwd(H_t, H_d, W, K, workspace=torch.empty(least_workspace(N, d, V, K), dtype=torch.uint8, device=dev))
    assert not torch.equal(a["dH_d"], b["dH_d"])      # (p from a bf16 spill or from fp32 logits: two routes)
    for out in (a, b):
        hass.check(out["workspace"])
        print(compare(inp.H_t, inp.H_d[0], inp.W, K, {k: v.cpu() for k, v in out.items() if k != "workspace"}))
    loss = torch.empty(N, dtype=torch.float32).pin_memory()
    dH = torch.empty(N, d, dtype=torch.bfloat16).pin_memory()
    hass.topk_distill_fwd_bwd_host(inp.H_t.pin_memory(), inp.H_d[0].pin_memory(), W, K, loss, dH)
    assert torch.equal(loss, a["loss"].cpu()) and torch.equal(dH, a["dH_d"].cpu())


@pytest.mark.parametrize("K", [10, 40])
def test_nan_logits_hide_no_candidate(K):
    """Tokens whose rows of W are NaN make a row's sums NaN, but the first tile's admission bound must not count them."""
    import paper_2408_15766_b200 as hass
    inp = hi.make_custom(64, 64, 1024, K, seed=4, sigma_w=0.3)
    W = inp.W.clone()
    W[16:48] = float("nan")
    W[200:230] = float("nan")
    dev = torch.device("cuda:0")
    out = hass.topk_distill_fwd(inp.H_t.to(dev), inp.H_d[0].to(dev), W.to(dev), K)
    hass.check(out["workspace"])
    z = (inp.H_t.double() @ W.double().T).nan_to_num(nan=-np.inf)
    want = z.topk(K, dim=1).indices.sort(dim=1).values
    assert torch.equal(out["topk_idx"].cpu().long().sort(dim=1).values, want)
