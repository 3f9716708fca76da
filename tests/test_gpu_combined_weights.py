"""Combined objective where target and draft are peaked on different tokens: the Top-K term w q of such a token is held in fp32."""
import numpy as np
import pytest
import torch

import hass_inputs as hi

pytestmark = pytest.mark.gpu


# A row's form: one block of 512, 256 or 128 threads or a cluster of blocks with the row in registers, one of 1024 or 512 threads that reads it
# twice; sets within the first warp and beyond it; chunks of as many row tiles as there is room for in fp32
@pytest.mark.parametrize("N,V,K", [(40, 1000, 10), (40, 2100, 40), (9, 30000, 10), (3, 9000, 200), (100, 32000, 10), (300, 1000, 10), (300, 2000, 40),
                                   (300, 9000, 10), (520, 9000, 33), (9345, 1000, 4)])
def test_the_target_s_token_keeps_its_weight(N, V, K):
    import paper_2408_15766_b200 as hass
    dev = torch.device("cuda:0")
    d, token, w = 72, 5, 8.0
    inp = hi.make_custom(N, d, V, K, seed=V + K, sigma_w=0.05)
    W, H_t, H_d = inp.W.clone(), inp.H_t.clone(), inp.H_d[0].clone()
    # feature 0: the target's favourite, far down in the draft; feature 1: of that token alone, so that dH_d's is dz_d of that token
    W[:, :2] = 0
    W[token, :2] = 1
    H_t[:, 0] = torch.as_tensor(np.random.default_rng(K).uniform(-1.0, 3.0, size=N) + np.log(V)).to(torch.bfloat16)
    H_d[:, 0] = -8
    H_t[:, 1] = H_d[:, 1] = 0
    out = hass.combined_distill_fwd_bwd(H_t.to(dev), H_d.to(dev), W.to(dev), K, w, dH_dtype=hass.HASS_FP32)
    hass.check(out["workspace"])
    z_t, z_d = (x.double() @ W.double().T for x in (H_t, H_d))
    q, p = z_t.softmax(1), z_d.softmax(1)
    want = (1 + w * q.topk(K, 1).values.sum(1)) * p[:, token] - (1 + w) * q[:, token]
    error = float(((out["dH_d"][:, 1].cpu().double() - want).abs() / want.abs()).max())
    print(f"{N} x {V}, K = {K}: {error:.2e}")
    # fp32 throughout: a logit's last bit (2^-20 of logits up to 14) in the exponent, and those of a sum of nine terms; one rounding to bf16 is up to 2^-8
    assert error < 1e-5
