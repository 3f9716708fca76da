"""The forms of the GEMM kernel at the sizes where they can go wrong: CTA pairs whose last row tile has no partner, output
tiles cut along the contraction (alone, behind whole rounds, with few rows), against the oracle with the tolerances of
the parity tests, every buffer between guard bands."""
import numpy as np
import pytest

import hass_inputs as hi
from parity import compare
from test_gpu_parity import _guarded_fused

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d,V,K,fp32", [
    (1600, 64, 5000, 10, True),        # 13 row tiles as seven pairs, the last one with a tile of its own only
    (1537, 200, 3000, 20, False),      # the same with one row in the last tile and a ragged last column tile
    (61, 520, 20000, 10, False),       # one row tile: cut output tiles that keep 61 rows
    (129, 264, 30001, 5, True),        # two row tiles, one row in the second, a ragged contraction
    (1601, 2824, 12000, 10, False),    # whole rounds of output tiles, then a cut rest, d not a multiple of 256
])
def test_pairs_and_cut_tiles(N, d, V, K, fp32):
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=2.0 / np.sqrt(d))
    grad = np.random.default_rng(1).normal(size=N)
    rows = None if N * d * V < 3e9 else np.unique(np.r_[0:8, 120:136, N - 70:N - 60, N - 8:N])
    fused, split = _guarded_fused(inp, K, grad, dH_fp32=fp32)
    print("fused", compare(inp.H_t, inp.H_d[0], inp.W, K, fused, grad_loss=grad, rows=rows))
    print("split", compare(inp.H_t, inp.H_d[0], inp.W, K, split, grad_loss=grad, rows=rows))
