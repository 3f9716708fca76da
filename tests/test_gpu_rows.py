"""Calls of at most 128 rows: the logits of both feature sets in fp32, one block per row for statistics, Top-K and dz_d."""
import numpy as np
import pytest
import torch

import hass_inputs as hi
import oracle
from parity import compare, compare_variant

pytestmark = pytest.mark.gpu


def _hass():
    import paper_2408_15766_b200 as hass
    return hass


def _cpu(out):
    return {k: v.cpu() for k, v in out.items() if k != "workspace"}


# fewer logits than threads, a thread's first piece and one logit more, a step of the pass and one logit more, all K tokens
@pytest.mark.parametrize("N,d,V,K", [(1, 64, 1024, 256), (3, 64, 300, 256), (5, 8, 9, 5), (7, 16, 4097, 128),
                                     (64, 64, 16384, 17), (65, 72, 16385, 100), (128, 64, 33000, 1), (33, 72, 1024, 64), (20, 64, 1024, 65)])
def test_rows_against_the_oracle(N, d, V, K):
    hass = _hass()
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=0.3)
    H_t, H_d, W = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev)
    g = np.random.default_rng(N).uniform(-1.0, 1.0, size=N)
    gd = torch.tensor(g, dtype=torch.float32, device=dev)
    out = hass.topk_distill_fwd_bwd(H_t, H_d, W, K, grad_loss=gd, dH_dtype=hass.HASS_FP32)
    hass.check(out["workspace"])
    print("fused", compare(inp.H_t, inp.H_d[0], inp.W, K, _cpu(out), grad_loss=g))
    draft = hass.topk_distill_fwd_bwd_draft(H_d, W, out["topk_idx"], out["topk_q"], grad_loss=gd, dH_dtype=hass.HASS_FP32)
    hass.check(draft["workspace"])
    for k in ("loss", "lse_d", "dH_d"):
        assert torch.equal(draft[k], out[k]), k
    fwd = hass.topk_distill_fwd(H_t, H_d, W, K)
    hass.check(fwd["workspace"])
    for k in ("loss", "lse_t", "lse_d", "topk_idx", "topk_q"):
        assert torch.equal(fwd[k], out[k]), k


@pytest.mark.parametrize("V,K,first", [(700, 40, 0), (5000, 1, 3000), (5000, 200, 1), (40000, 256, 17)])
def test_equal_logits_give_the_lowest_tokens(V, K, first):
    """From token `first` on all rows of W are the same, the others' logits lie below: more equal logits than the pool holds."""
    hass = _hass()
    dev = torch.device("cuda:0")
    d = 64
    H = torch.ones(3, d, dtype=torch.bfloat16, device=dev)
    W = torch.full((V, d), 0.125, dtype=torch.bfloat16, device=dev)
    W[:first] = -0.125
    out = hass.topk_distill_fwd_bwd(H, H, W, K)
    hass.check(out["workspace"])
    assert torch.equal(out["topk_idx"].cpu().long(), torch.arange(first, first + K).expand(3, K))


@pytest.mark.parametrize("N,d,V,K", [(1, 264, 8200, 20), (64, 512, 4100, 7), (100, 264, 8200, 128), (128, 8, 270000, 3)])
def test_variants_of_few_rows_against_the_oracle(N, d, V, K):
    """The Omega_hat term of the Bi-directional variant stays in fp32 on this route too."""
    hass = _hass()
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=0.1)
    args = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev), K
    for variant, which, param in ((hass.LOSS_BIDIR_TOPK, oracle.VARIANT_BIDIR, 0.0), (hass.LOSS_NORMED_TOPK, oracle.VARIANT_NORMED, 0.0),
                                  (hass.LOSS_TOP_P, oracle.VARIANT_TOP_P, 0.002)):
        if which == oracle.VARIANT_NORMED and K == 1:
            continue
        out = hass.variant_distill_fwd_bwd(*args, variant, param, dH_dtype=hass.HASS_FP32)
        hass.check(out["workspace"])
        print(which, compare_variant(inp.H_t, inp.H_d[0], inp.W, K, which, param, _cpu(out)))


# One, two, four and eight blocks per row and one logit more, as many rows as their blocks are resident for and one more (a block
# per row), a last block with a piece of one logit, with none, and rows longer than eight blocks take
@pytest.mark.parametrize("N,d,V,K", [(1, 64, 8192, 256), (74, 16, 8193, 100), (75, 16, 8193, 100), (37, 64, 16385, 10), (2, 64, 24577, 33),
                                     (18, 8, 32769, 64), (19, 8, 65537, 64), (2, 16, 131072, 128), (2, 16, 131073, 10)])
def test_rows_split_over_blocks_against_the_oracle(N, d, V, K):
    hass = _hass()
    dev = torch.device("cuda:0")
    inp = hi.make_custom(N, d, V, K, seed=N + V, sigma_w=0.3)
    args = inp.H_t.to(dev), inp.H_d[0].to(dev), inp.W.to(dev), K
    out = hass.topk_distill_fwd_bwd(*args, dH_dtype=hass.HASS_FP32)
    hass.check(out["workspace"])
    print("fused", compare(inp.H_t, inp.H_d[0], inp.W, K, _cpu(out)))
    for variant, which in ((hass.LOSS_NORMED_TOPK, oracle.VARIANT_NORMED), (hass.LOSS_BIDIR_TOPK, oracle.VARIANT_BIDIR)):
        if which == oracle.VARIANT_BIDIR and K > 128:
            continue
        out = hass.variant_distill_fwd_bwd(*args, variant, dH_dtype=hass.HASS_FP32)
        hass.check(out["workspace"])
        print(which, compare_variant(inp.H_t, inp.H_d[0], inp.W, K, which, 0.0, _cpu(out)))


# A row of one block, of two blocks, the row kernel, and the separate backward of more rows
@pytest.mark.parametrize("N,V", [(5, 600), (5, 20000), (100, 9000), (200, 600)])
def test_backward_of_a_set_that_repeats_a_token(N, V):
    """The separate backward takes any set: a token named twice has both of its probabilities taken off, a cut entry (-1) none."""
    hass = _hass()
    dev = torch.device("cuda:0")
    d, K = 64, 12
    g = torch.Generator().manual_seed(V)
    H, W = torch.randn(N, d, generator=g).to(torch.bfloat16), (0.3 * torch.randn(V, d, generator=g)).to(torch.bfloat16)
    idx = torch.randint(0, V, (N, K), generator=g, dtype=torch.int32)
    idx[:, 7], idx[:, 9], idx[1:, 3] = idx[:, 2], idx[:, 2], idx[1:, 11]
    q = torch.rand(N, K, generator=g) / K
    q[::2, 2] = 0.0
    idx[:, 5], q[:, 5] = -1, 0.0
    z = H.double() @ W.double().T
    lse = z.logsumexp(1)
    dz = q.double().sum(1, keepdim=True) * (z - lse[:, None]).exp()
    dz.scatter_add_(1, idx.clamp(min=0).long(), -q.double())
    want = dz @ W.double()
    ws = torch.empty(hass.topk_distill_workspace_bytes(N, d, V, K), dtype=torch.uint8, device=dev)
    dH = hass.topk_distill_bwd(H.to(dev), W.to(dev), idx.to(dev), q.to(dev), lse.float().to(dev), dH_dtype=hass.HASS_FP32, workspace=ws)
    hass.check(ws)
    # every entry of dz_d in bf16, 2^-9 of itself
    assert (dH.cpu().double() - want).abs().max() <= 1e-2 * want.abs().max()


# 40 rows: the row kernel; 200: the spill and its patch. A vocabulary masked by a bias column of -inf, so that fewer than K tokens
# are left: token 0 with q = 0 fills the set up, whether it is one of those left or not.
@pytest.mark.parametrize("N,V", [(40, 700), (200, 30)])
@pytest.mark.parametrize("K", [10, 20])
@pytest.mark.parametrize("left", [(0, 3, 7, 11, 12, 29), (5, 6, 17, 28)])
def test_fewer_than_k_tokens_above_minus_infinity(N, V, K, left):
    hass = _hass()
    d = 64
    inp = hi.make_custom(N, d, V, K, seed=N + K, sigma_w=0.5)
    H_t, H_d, W = inp.H_t.clone(), inp.H_d[0].clone(), inp.W.clone()
    H_t[:, 0] = H_d[:, 0] = 1.0
    masked = torch.ones(V, dtype=torch.bool)
    masked[list(left)] = False
    W[masked, 0] = -float("inf")
    z_t, z_d = ((H[:, 1:].double() @ W[:, 1:].double().T + (H[:, :1].double() @ W[:, :1].double().T)).masked_fill(masked, -np.inf) for H in (H_t, H_d))
    q, idx = z_t.softmax(1).topk(len(left), dim=1)
    log_p = z_d.log_softmax(1)
    dz = q.sum(1, keepdim=True) * log_p.exp()
    dz.scatter_add_(1, idx, -q)
    want = {"loss": -(q * log_p.gather(1, idx)).sum(1), "lse_t": z_t.logsumexp(1), "lse_d": z_d.logsumexp(1), "dH_d": dz @ W[:, 1:].double()}
    dev = torch.device("cuda:0")
    args = H_t.to(dev), H_d.to(dev), W.to(dev), K
    out = hass.topk_distill_fwd_bwd(*args, dH_dtype=hass.HASS_FP32)
    hass.check(out["workspace"])
    draft = hass.topk_distill_fwd_bwd_draft(args[1], args[2], out["topk_idx"], out["topk_q"], dH_dtype=hass.HASS_FP32)
    hass.check(draft["workspace"])
    assert torch.equal(out["topk_idx"].cpu()[:, :len(left)].long(), idx)
    assert (out["topk_idx"].cpu()[:, len(left):] == 0).all() and (out["topk_q"].cpu()[:, len(left):] == 0).all()
    for got in (_cpu(out), _cpu(draft)):
        for k in ("loss", "lse_t", "lse_d"):
            # fp32 sums of 64 products of up to 8, as in the parity tests
            assert k not in got or (got[k].double() - want[k]).abs().max() <= 1e-4, k
        # (column 0: the weights of the masked tokens are zero times -inf) dz_d in bf16, 2^-9 of its largest entry or so
        err = (got["dH_d"][:, 1:].double() - want["dH_d"]).abs().max()
        assert err <= 1e-2 * want["dH_d"].abs().max()


def _levels(V, pattern):
    """Logits of a vocabulary at which the bound from the threads' maxima (thread (v // 4) % 1024 owns token v) admits more than the
    pool holds: three digits of up to eight bits each, so that every sum below is exact."""
    v = torch.arange(V)
    owner = v // 4 % 1024
    if pattern == "few above":            # 41 distinct logits above a level that all others share
        hi = torch.where(v % 977 == 5, 2.0, 1.0)
        return hi, torch.where(v % 977 == 5, (v // 977) / 64.0, torch.zeros(V))
    if pattern == "by thread":            # what a thread owns lies close together, the threads apart; nearly no ties
        return (owner // 16).float(), owner % 16 / 16.0 + v % 4 / 128.0 + (v // 4096) / 1024.0 % 0.0078125
    if pattern == "two levels":           # the largest logit five times in all, then every second token alike
        return torch.where(v % 8000 == 4001, 3.0, 1.0), (v % 2) / 2.0
    hi = torch.where(owner % 10 == 3, 1.0, -float("inf"))      # "masked": a tenth of the threads has all there is
    return hi, v % 61 / 64.0


@pytest.mark.parametrize("K", [1, 64, 256])
@pytest.mark.parametrize("pattern", ["few above", "by thread", "two levels", "masked"])
def test_more_logits_at_the_bound_than_the_pool_holds(pattern, K):
    hass = _hass()
    dev = torch.device("cuda:0")
    V, d = 40001, 64
    W = torch.zeros(V, d, dtype=torch.bfloat16)
    hi, lo = _levels(V, pattern)
    W[:, 0] = hi.to(torch.bfloat16)
    W[:, 1] = lo.to(torch.bfloat16)
    W[:, 2] = (lo - lo.to(torch.bfloat16).float()).to(torch.bfloat16)
    H = torch.zeros(2, d, dtype=torch.bfloat16)
    H[:, :3] = 1.0
    H[1, 1:] = 0.0                        # the second row has the first digit alone: ties everywhere
    z = H[:, 1:].double() @ W[:, 1:].double().T + W[:, 0].double()
    want = z.sort(dim=1, descending=True, stable=True).indices[:, :K]
    out = hass.topk_distill_fwd(H.to(dev), H.to(dev), W.to(dev), K)
    hass.check(out["workspace"])
    assert torch.equal(out["topk_idx"].cpu().long(), want)


@pytest.mark.parametrize("d,V,K", [(256, 128256, 10), (256, 128256, 64), (256, 1024, 10)])
def test_rows_of_zeros_take_no_longer(d, V, K):
    """Feature rows of zeros (padding) have V equal logits. Where token ids are searched bit by bit, they take a call of 128256 tokens
    from 107 to 874 us, and ranking 1024 equal logits one of 1024 from 42 to 97; with one look at the first tokens neither changes."""
    hass = _hass()
    dev = torch.device("cuda:0")
    inp = hi.make_custom(8, d, V, K, seed=1, sigma_w=0.05)
    W = inp.W.to(dev)
    ws = torch.empty(hass.topk_distill_workspace_bytes(8, d, V, K), dtype=torch.uint8, device=dev)
    features = []
    for zero in (False, True):
        H_t, H_d = inp.H_t.clone(), inp.H_d[0].clone()
        if zero:
            H_t[4:] = 0
            H_d[4:] = 0
        features.append((H_t.to(dev), H_d.to(dev)))
    times = [[], []]
    for i in range(120):      # (in turn, and the least of each: the host is part of these calls' time)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        hass.topk_distill_fwd_bwd(*features[i % 2], W, K, workspace=ws)
        b.record()
        b.synchronize()
        times[i % 2].append(a.elapsed_time(b) * 1e3)
    hass.check(ws)
    plain, zeros = (min(t[5:]) for t in times)
    print(plain, zeros)
    assert zeros <= 1.25 * plain + 20.0


@pytest.mark.parametrize("V,K", [(700, 5), (5000, 40)])
def test_an_infinite_logit_comes_first(V, K):
    hass = _hass()
    dev = torch.device("cuda:0")
    inp = hi.make_custom(3, 64, V, K, seed=V, sigma_w=0.3)
    H, W = inp.H_t.clone(), inp.W.clone()
    H[:, 0] = 1.0
    W[[V - 3, 17], 0] = float("inf")
    W[300:400, 0] = -float("inf")
    out = hass.topk_distill_fwd(H.to(dev), H.to(dev), W.to(dev), K)
    hass.check(out["workspace"])
    z = H[:, 1:].double() @ W[:, 1:].double().T + W[:, 0].double()
    assert torch.equal(out["topk_idx"].cpu().long(), z.sort(dim=1, descending=True, stable=True).indices[:, :K])
