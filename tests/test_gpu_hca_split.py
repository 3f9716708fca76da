"""Backward of the HCA attention with every key tile's work in two halves, where few key tiles would leave SMs idle."""
import pytest
import torch

import hass_inputs as hi

pytestmark = pytest.mark.gpu


# Split on 148 SMs: a last key tile of one position (a single element: an empty half) and odd halves, with and without draft passes and
# with a key/value head for every query head; odd halves of a group of three; more halves than SMs, so that a CTA takes several. Not
# split (the longest item does not get a fifth shorter): the same tests hold.
@pytest.mark.parametrize("B,T,H,Hkv,m,split", [(1, 1025, 1, 1, 0, True), (1, 2049, 1, 1, 1, True), (1, 2049, 2, 2, 8, True), (1, 700, 3, 1, 1, True),
                                               (2, 1100, 32, 8, 2, True), (1, 129, 1, 1, 0, False), (2, 333, 4, 2, 3, False),
                                               (1, 1025, 16, 16, 8, False)])
def test_halves_of_a_key_tile_add_up_to_the_whole(B, T, H, Hkv, m, split):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    inp = hi.make_hca_inputs(hi.HcaWorkload("split", B=B, T=T, H=H, Hkv=Hkv, m=m, seed=T))
    dO = torch.randn(inp.Q.shape, generator=torch.Generator().manual_seed(1)).to(torch.bfloat16).to(dev)
    qkv = [x.to(dev) for x in (inp.Q, inp.K_t, inp.V_t)]
    Kd, Vd = [x.to(dev) for x in inp.K_d], [x.to(dev) for x in inp.V_d]
    fw = hass.hca_attention_fwd(*qkv, Kd, Vd)
    hass.check(fw["workspace"])
    whole = 256 + -(-B * H * T * 4 // 256) * 256 + B * T * H * 512      # status, D, the dQ accumulator: no room for the halves
    full = hass.hca_attention_bwd_workspace_bytes(B, T, H, m)
    assert full > whole
    runs = []
    for size in (whole, full, full):
        ws = torch.full((size,), 0xAB, dtype=torch.uint8, device=dev)
        bw = hass.hca_attention_bwd(*qkv, Kd, Vd, fw["O"], fw["lse"], dO, workspace=ws)
        hass.check(bw["workspace"])
        runs.append(bw)
        # the halves' fp32 dV and dK lie behind the rest
        assert bool((ws[whole:] != 0xAB).any()) == (split and size == full)
    for name in ("dQ", "dK_t", "dV_t"):
        a, b = runs[0][name].float(), runs[1][name].float()
        # fp32 sums in another order, rounded to bf16: one unit in the last place (2^-7 of the value), or 1e-5 of the largest
        # entry where a sum cancels
        assert ((a - b).abs() <= 2.0 ** -7 * a.abs() + 1e-5 * a.abs().max()).all(), name
    for name in ("dK_t", "dV_t"):
        assert torch.equal(runs[1][name], runs[2][name]), name
