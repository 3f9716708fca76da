"""Calls of at most 128 rows choose what the L2 holds of W between its two readings: nothing of that outlasts the call."""
import pytest
import torch

import hass_inputs as hi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", ["fwd_bwd", "fwd"])
def test_the_caller_s_data_has_the_l2_again_after_a_call(which):
    """80 MB that the caller walks over fit the L2; with 64 MB of W held in it, each pass over them took 26.6 us instead of 21.5."""
    import paper_2408_15766_b200 as hass
    N, d, V, K = 8, 4096, 32000, 10
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(1)
    H = torch.randn(N, d, generator=g, device=dev).to(torch.bfloat16)
    W = torch.randn(V, d, generator=g, device=dev).mul_(0.02).to(torch.bfloat16)
    ws = torch.empty(hass.topk_distill_workspace_bytes(N, d, V, K), dtype=torch.uint8, device=dev)
    own = torch.zeros(80 << 18, dtype=torch.float32, device=dev)

    def pass_us():
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(13)]
        ev[0].record()
        for e in ev[1:]:
            own.mul_(1.0)
            e.record()
        torch.cuda.synchronize()
        return sorted(a.elapsed_time(b) * 1e3 for a, b in zip(ev[2:], ev[3:]))[5]      # (the first two bring the data back)

    for _ in range(3):
        before = pass_us()
    after = []
    for _ in range(5):
        if which == "fwd":
            hass.topk_distill_fwd(H, H, W, K, workspace=ws)
        else:
            hass.topk_distill_fwd_bwd(H, H, W, K, workspace=ws)
        after.append(pass_us())
    hass.check(ws)
    print(before, after)
    assert min(after) <= 1.08 * before + 0.5
