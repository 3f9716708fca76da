"""Top-K sets of more than 16 tokens: what the lanes of a row tile tell one another about the row, on vocabularies whose large
logits are spread evenly, lie in one lane's column tiles, come late, come early, or are all alike."""
import pytest
import torch

import hass_inputs as hi
from parity import compare

pytestmark = pytest.mark.gpu


def _shared_bounds(ws, N, V, K):
    """Whether lanes have shared their bounds in this workspace of the forward: the room behind the largest logits is not zero."""
    import paper_2408_15766_b200 as hass
    up = lambda x: -(-x // 256) * 256
    at = hass.topk_distill_fwd_static_scratch_bytes(N, 64, V, K) + 3 * up(N * K * 4) + 2 * up(N * 4) + 2 * -(-N // 128) * 128 * 4
    return bool(ws[at:at + 128 * 8].view(torch.int32).any())


# On 148 SMs: lanes of one column tile; of one or two; of two or three (125 tiles on 49 lanes), a pair per row tile; of six or seven (50 on
# 8), the last row tile alone in its pair; of three (24 on 8). From three tiles on lanes share their bounds.
@pytest.mark.parametrize("N,V,shared", [(300, 6000, False), (300, 12800, False), (300, 32000, True), (2100, 12800, True), (2100, 6000, True)])
@pytest.mark.parametrize("K", [17, 100, 256])
@pytest.mark.parametrize("layout", ["even", "one tile", "rising", "falling", "alike"])
def test_sets_of_large_k(N, V, shared, K, layout):
    import paper_2408_15766_b200 as hass
    d = 64
    inp = hi.make_custom(N, d, V, K, seed=V + K, sigma_w=0.3)
    H_t, W = inp.H_t.clone(), inp.W.clone()
    H_t[:, 0] = 4.0
    at = torch.arange(V, dtype=torch.float32) / V
    if layout == "one tile":
        W[256:512, 0] = 2.0
    elif layout == "rising":
        W[:, 0] = (2.0 * at).to(torch.bfloat16)
    elif layout == "falling":
        W[:, 0] = (-2.0 * at).to(torch.bfloat16)
    elif layout == "alike":
        H_t[:, 1:] = 0.0
        W[:, 0] = (torch.arange(V) % 3).to(torch.bfloat16)      # three values: a third of the vocabulary ties at the top
    dev = torch.device("cuda:0")
    ws = torch.zeros(hass.topk_distill_workspace_bytes(N, d, V, K), dtype=torch.uint8, device=dev)
    out = hass.topk_distill_fwd(H_t.to(dev), inp.H_d[0].to(dev), W.to(dev), K, workspace=ws)
    hass.check(ws)
    assert _shared_bounds(ws, N, V, K) == shared
    cpu = {k: v.cpu() for k, v in out.items() if k != "workspace"}
    if layout == "alike":
        assert torch.equal(cpu["topk_idx"].long(), (2 + 3 * torch.arange(K)).expand(N, K))
    else:
        want = (H_t.double() @ W.double().T).topk(K, dim=1).values
        z = (H_t.double() @ W.double().T).gather(1, cpu["topk_idx"].long())
        assert (z - want).abs().max() <= 1e-4      # fp32 sums of 64 products of up to 8 in another order: 64 x 2^-24 x 16
        print(compare(H_t, inp.H_d[0], W, K, cpu, check_dH=False, rows=range(0, N, 37)))


@pytest.mark.parametrize("K", [17, 100])
def test_the_least_workspace_gives_the_same_sets(K):
    """Lanes share their bounds in room that the call does not use meanwhile; a workspace that ends before it does without."""
    import paper_2408_15766_b200 as hass
    N, d, V = 2100, 64, 12800
    inp = hi.make_custom(N, d, V, K, seed=K, sigma_w=0.3)
    dev = torch.device("cuda:0")
    args = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev), K
    least = torch.empty(hass.topk_distill_fwd_static_scratch_bytes(N, d, V, K), dtype=torch.uint8, device=dev)
    a, b = hass.topk_distill_fwd(*args, workspace=least), hass.topk_distill_fwd(*args)
    hass.check(a["workspace"])
    hass.check(b["workspace"])
    assert torch.equal(a["topk_idx"], b["topk_idx"])
