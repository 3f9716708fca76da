"""Performance cases of the fused LM-head + Top-K distillation loss and of the HCA attention.

Every case is one step as a draft-head trainer takes it, through the package's public functions, on device tensors
that the trainer holds anyway: features of one batch, the frozen LM head, a workspace kept between steps. The sizes
are the workloads of this repository (LLaMA2-7B/13B and LLaMA3-8B/70B heads, the tiny configuration, the two HCA
geometries), full batches and the shorter, ragged ones that the end of an epoch or short conversations give.

ops
  fwd_bwd        topk_distill_fwd_bwd: loss and gradient of the first aligning step
  fwd_bwd_draft  topk_distill_fwd_bwd_draft: the same for the later aligning steps, which reuse the target's Top-K set
  split          topk_distill_fwd, then topk_distill_bwd: what an autograd function calls
  combined       combined_distill_fwd_bwd: cross-entropy plus the weighted Top-K loss
  top_p, normed, bidir   variant_distill_fwd_bwd: the loss variants
  hca            hca_attention_fwd and, with "bwd", hca_attention_bwd: the attention of the draft layer
"""
from __future__ import annotations

import math

import torch

import paper_2408_15766_b200 as hass

# (d, V, standard deviation of W): the LM heads of the target models, and the tiny configuration
HEADS = {
    "tiny": (256, 1024, 0.02),
    "l2-7b": (4096, 32000, 0.02),
    "l2-13b": (5120, 32000, 0.02),
    "l3-8b": (4096, 128256, 0.02),
    "l3-70b": (8192, 128256, 0.015),
}
# (query heads, key/value heads) of the draft layer; head dimension 128
ATTENTION = {"tiny": (2, 1), "mid": (4, 2), "l2-7b": (32, 32), "l2-13b": (40, 40), "l3-8b": (32, 8), "l3-70b": (64, 8)}
HEAD_DIM = 128
VARIANTS = {"top_p": hass.LOSS_TOP_P, "normed": hass.LOSS_NORMED_TOPK, "bidir": hass.LOSS_BIDIR_TOPK}


def _loss_case(op, N, d, V, K, sigma=0.02, fp32=False, weights=False, name=None):
    c = {"op": op, "N": N, "d": d, "V": V, "K": K, "sigma": sigma, "fp32": fp32, "weights": weights}
    if name:
        c["name"] = name
    return c


def _head_case(op, head, N, K, name, **kw):
    d, V, sigma = HEADS[head]
    return _loss_case(op, N, d, V, K, sigma, name=name, **kw)


def _hca_case(B, T, H, Hkv, m, bwd, name=None):
    c = {"op": "hca", "B": B, "T": T, "H": H, "Hkv": Hkv, "m": m, "bwd": bwd}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a unit test's or a sanity run's step, all latency
        _head_case("fwd_bwd", "tiny", 64, 10, "tiny", fp32=True),
        # one short conversation through a real head: bound by reading W
        _head_case("fwd_bwd", "l2-7b", 61, 10, "l2-7b-short"),
        # a ragged batch of a few short sequences with per-position weights (padding masked by zeros)
        _head_case("fwd_bwd", "l3-8b", 517, 10, "l3-8b-ragged", weights=True),
        # full batches of 8192 positions: the configurations the framework is quoted on
        _head_case("fwd_bwd", "l2-7b", 8192, 10, "l2-7b"),
        _head_case("fwd_bwd_draft", "l2-13b", 8192, 10, "l2-13b-draft"),
        _head_case("fwd_bwd", "l3-8b", 8192, 10, "l3-8b"),
        # the largest head, with a large Top-K set
        _head_case("fwd_bwd", "l3-70b", 4096, 64, "l3-70b-k64"),
        # forward and backward as two calls (autograd), the largest K of the paper's sweep, fp32 gradient
        _head_case("split", "l2-7b", 2047, 100, "l2-7b-split-k100", fp32=True),
        # the whole training objective of an aligning step on one 1024-token sequence
        _head_case("combined", "l3-8b", 1024, 10, "l3-8b-combined"),
        # the heaviest of the loss variants on one 2048-token sequence
        _head_case("bidir", "l2-7b", 2048, 10, "l2-7b-bidir"),
        # the draft layer's attention in the third aligning step, forward and backward: the full batch ...
        _hca_case(4, 2048, *ATTENTION["l3-8b"], 2, True, "hca-l3-8b"),
        # ... and a short ragged one
        _hca_case(2, 333, *ATTENTION["mid"], 3, True, "hca-mid"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MAX_MACS = 3.0 * 8192 * 4096 * 128256     # three products of the largest listed step


def draw(rng):
    if rng.random() < 0.25:
        H, Hkv = ATTENTION[rng.choice(sorted(ATTENTION))]
        T = _log_int(rng, 16, 4096)
        B = rng.randint(1, max(1, min(8, 8192 // T)))
        return _hca_case(B, T, H, Hkv, rng.randint(0, 5), rng.random() < 0.7)
    op = rng.choice(["fwd_bwd", "fwd_bwd", "fwd_bwd_draft", "split", "combined", "top_p", "normed", "bidir"])
    if rng.random() < 0.7:
        d, V, sigma = HEADS[rng.choice(sorted(HEADS))]
    else:
        d, V, sigma = 8 * _log_int(rng, 32, 1024), _log_int(rng, 1000, 130000), 0.02
    N = _log_int(rng, 1, 8192)
    N = max(1, min(N, int(MAX_MACS * 0.7 / (4.0 * d * V))))
    # (Normed Top-K over a single token is constant: no loss and no gradient)
    K = _log_int(rng, 2 if op == "normed" else 1, 64 if op == "bidir" else 128)
    return _loss_case(op, N, d, V, K, sigma, fp32=rng.random() < 0.25, weights=rng.random() < 0.3)


def _randn(g, shape, std=1.0):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).mul_(std)


def _bf16_randn(g, rows, cols, std):
    """Drawn in pieces, so that the fp32 values of a large head are never held at once."""
    out = torch.empty(rows, cols, dtype=torch.bfloat16, device="cuda")
    step = max(1, (1 << 26) // cols)
    for r in range(0, rows, step):
        n = min(step, rows - r)
        out[r:r + n] = _randn(g, (n, cols), std)
    return out


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["op"] == "hca":
        return _prepare_hca(case, g)
    N, d, V, K, op = case["N"], case["d"], case["V"], case["K"], case["op"]
    dtype = hass.HASS_FP32 if case["fp32"] else hass.HASS_BF16
    H_t = _randn(g, (N, d))
    H_d = (H_t + _randn(g, (N, d), 0.5)).to(torch.bfloat16)
    s = {"op": op, "K": K, "dtype": dtype, "H_t": H_t.to(torch.bfloat16), "H_d": H_d, "W": _bf16_randn(g, V, d, case["sigma"]),
         "grad": None}
    if case["weights"]:
        # the aligning step's weight over the number of positions, and one position in eight masked
        w = torch.rand(N, generator=g, device="cuda")
        s["grad"] = torch.where(w < 0.125, torch.zeros_like(w), torch.full_like(w, 1.0)).mul_(1.0 / N)
    if op == "combined":
        nbytes = hass.combined_distill_workspace_bytes(N, d, V, K)
    else:
        nbytes = hass.topk_distill_workspace_bytes(N, d, V, K)
    s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    if op == "fwd_bwd_draft":
        # the target's Top-K set and probabilities, as the first aligning step left them
        first = hass.topk_distill_fwd(s["H_t"], s["H_d"], s["W"], K, workspace=s["ws"])
        s["topk_idx"], s["topk_q"] = first["topk_idx"], first["topk_q"]
    if op == "top_p":
        # P at which the prefixes of these near-uniform rows are a few dozen tokens, as many as K at most
        s["p"] = 0.01
    return s


def _prepare_hca(case, g):
    B, T, H, Hkv, m = case["B"], case["T"], case["H"], case["Hkv"], case["m"]
    kv = (B, T, Hkv, HEAD_DIM)
    K, V = _randn(g, kv), _randn(g, kv)
    s = {"op": "hca", "bwd": case["bwd"], "Q": _randn(g, (B, T, H, HEAD_DIM)).to(torch.bfloat16),
         "K_t": K.to(torch.bfloat16), "V_t": V.to(torch.bfloat16),
         "K_d": [(K + _randn(g, kv, 0.5)).to(torch.bfloat16) for _ in range(m)],
         "V_d": [(V + _randn(g, kv, 0.5)).to(torch.bfloat16) for _ in range(m)],
         "ws": torch.empty(hass.hca_attention_workspace_bytes(), dtype=torch.uint8, device="cuda")}
    if case["bwd"]:
        s["dO"] = _randn(g, (B, T, H, HEAD_DIM)).to(torch.bfloat16)
        s["ws_bwd"] = torch.empty(hass.hca_attention_bwd_workspace_bytes(B, T, H, m), dtype=torch.uint8, device="cuda")
    return s


def _results(*outs):
    """All tensors a call wrote, without the workspace."""
    got = {}
    for out in outs:
        got.update((k, v) for k, v in out.items() if k != "workspace")
    return got


def run(s):
    op = s["op"]
    if op == "hca":
        fwd = hass.hca_attention_fwd(s["Q"], s["K_t"], s["V_t"], s["K_d"], s["V_d"], workspace=s["ws"])
        if not s["bwd"]:
            return _results(fwd)
        bwd = hass.hca_attention_bwd(s["Q"], s["K_t"], s["V_t"], s["K_d"], s["V_d"], fwd["O"], fwd["lse"], s["dO"],
                                     workspace=s["ws_bwd"])
        return _results(fwd, bwd)
    if op == "fwd_bwd":
        return _results(hass.topk_distill_fwd_bwd(s["H_t"], s["H_d"], s["W"], s["K"], grad_loss=s["grad"],
                                                  dH_dtype=s["dtype"], workspace=s["ws"]))
    if op == "fwd_bwd_draft":
        return _results(hass.topk_distill_fwd_bwd_draft(s["H_d"], s["W"], s["topk_idx"], s["topk_q"], grad_loss=s["grad"],
                                                        dH_dtype=s["dtype"], workspace=s["ws"]))
    if op == "split":
        f = hass.topk_distill_fwd(s["H_t"], s["H_d"], s["W"], s["K"], workspace=s["ws"])
        dH = hass.topk_distill_bwd(s["H_d"], s["W"], f["topk_idx"], f["topk_q"], f["lse_d"], grad_loss=s["grad"],
                                   dH_dtype=s["dtype"], workspace=s["ws"])
        return dict(_results(f), dH_d=dH)
    if op == "combined":
        return _results(hass.combined_distill_fwd_bwd(s["H_t"], s["H_d"], s["W"], s["K"], w_topk=1.0, grad_loss=s["grad"],
                                                      dH_dtype=s["dtype"], workspace=s["ws"]))
    return _results(hass.variant_distill_fwd_bwd(s["H_t"], s["H_d"], s["W"], s["K"], VARIANTS[op], param=s.get("p", 0.0),
                                                 grad_loss=s["grad"], dH_dtype=s["dtype"], workspace=s["ws"]))


def work(case):
    """Products and tensors a step cannot do without: logits of both feature sets (the draft's alone when the Top-K set
    is given) and the gradient's back-projection; the combined objective also projects q. Normed Top-K needs the draft
    logits and the gradient on the K tokens only."""
    if case["op"] == "hca":
        B, T, H, Hkv, m = case["B"], case["T"], case["H"], case["Hkv"], case["m"]
        pairs = B * H * (T * (T + 1) // 2)
        q, kv = 2 * B * T * H * HEAD_DIM, 2 * B * T * Hkv * HEAD_DIM
        nbytes = 2 * q + (2 + 2 * m) * kv + 4 * B * H * T
        flops = 2 * 2 * HEAD_DIM * pairs
        if case["bwd"]:
            nbytes += 2 * q + (2 + 2 * m) * kv        # dO in; dQ and the gradients of keys and values out
            flops += 5 * 2 * HEAD_DIM * pairs
        return {"bytes": nbytes, "flops": flops}
    N, d, V, K, op = case["N"], case["d"], case["V"], case["K"], case["op"]
    products = {"fwd_bwd_draft": 2, "combined": 4, "normed": 1}.get(op, 3)
    features = 1 if op == "fwd_bwd_draft" else 2
    nbytes = 2 * V * d + 2 * N * d * features + (4 if case["fp32"] else 2) * N * d + 8 * N * K + 16 * N
    flops = 2 * products * N * d * V + (4 * N * K * d if op == "normed" else 0)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Four times what the outputs differ by from a float64 restatement of the same step. Gradients and attention outputs
    carry the rounding of bf16 weights and results (2-norm 1.6e-3 .. 3.3e-3; 5.9e-3 for the combined objective on small
    heads, where two bf16 projections nearly cancel). Two logits of the target that agree to fp32 rounding may swap ranks
    (3e-4 .. 5e-4 of the tokens at K >= 64), and where they swap at rank K one row's gradient moves (largest single
    difference 0.29 .. 0.57 of the root mean square)."""
    if case["op"] == "hca":
        return {"rel": 1.2e-2, "max": 0.35}
    return {"rel": 2.4e-2 if case["op"] == "combined" else 1.2e-2, "max": 0.8, "differ": 2e-3}


def exact(case, seed):
    """What run() returns for these inputs, in float64 torch; None for token ids, counts and values that a variant leaves out."""
    s = prepare(case, seed)
    return _exact_hca(s) if case["op"] == "hca" else _exact_loss(case, s)


def _exact_loss(case, s):
    op, K, N = case["op"], case["K"], case["N"]
    W = s["W"].double()
    rows = max(1, min(N, (1 << 27) // W.shape[0]))
    parts = []
    for r in range(0, N, rows):
        parts.append(_exact_rows(op, K, W, s, slice(r, min(N, r + rows))))
    got = {k: None if parts[0][k] is None else torch.cat([p[k] for p in parts]) for k in parts[0]}
    keys = {"fwd_bwd_draft": ("loss", "lse_d", "dH_d"), "combined": ("loss_ce", "loss", "topk_idx", "topk_q", "lse_t", "lse_d", "dH_d")}
    plain = ("loss", "topk_idx", "topk_q", "lse_t", "lse_d", "dH_d")
    variant = ("loss", "topk_idx", "topk_q", "topk_n", "lse_t", "lse_d", "dH_d")
    return {k: got[k] for k in keys.get(op, variant if op in VARIANTS else plain)}


def _exact_rows(op, K, W, s, rows):
    out = dict.fromkeys(("loss_ce", "topk_idx", "topk_q", "topk_n", "lse_t"))
    H_d = s["H_d"][rows].double()
    z_d = H_d @ W.T
    lse_d = z_d.logsumexp(1)
    p = (z_d - lse_d[:, None]).exp()
    g = s["grad"][rows].double()[:, None] if s["grad"] is not None else 1.0
    if op == "fwd_bwd_draft":
        idx, q = s["topk_idx"][rows].long(), s["topk_q"][rows].double()
        q_all = None
    else:
        z_t = s["H_t"][rows].double() @ W.T
        out["lse_t"] = z_t.logsumexp(1)
        q_all = (z_t - out["lse_t"][:, None]).exp()
        q, idx = q_all.topk(K, dim=1)
        if op == "top_p":
            q = torch.where(q.cumsum(1) - q > s["p"], 0.0, q)
        if op == "bidir":
            # the draft's K most probable tokens that the target's set does not hold, in descending p, then zeros
            idx_d = p.topk(K, dim=1).indices
            new = torch.ones_like(p, dtype=torch.bool).scatter_(1, idx, False).gather(1, idx_d)
            order = (~new).int().argsort(dim=1, stable=True)
            idx = torch.cat((idx, idx_d.gather(1, order)), 1)
            q = torch.cat((q, torch.where(new, q_all.gather(1, idx_d), 0.0).gather(1, order)), 1)
        out["topk_q"] = q
    if op == "normed":
        qn = q / q.sum(1, keepdim=True)
        zk = z_d.gather(1, idx)
        log_pn = zk.log_softmax(1)
        dz = torch.zeros_like(p).scatter_(1, idx, g * (log_pn.exp() - qn))
        return dict(out, loss=-(qn * log_pn).sum(1), lse_d=None, dH_d=dz @ W)
    log_p = z_d.gather(1, idx) - lse_d[:, None]
    if op == "combined":
        out["loss_ce"] = lse_d - (q_all * z_d).sum(1)
        dz = (1.0 + q.sum(1, keepdim=True)) * p - q_all
    else:
        dz = q.sum(1, keepdim=True) * p
    # (tokens beyond a variant's set carry q = 0)
    dz.scatter_add_(1, idx, -q)
    return dict(out, loss=-(q * log_p).sum(1), lse_d=lse_d, dH_d=(g * dz) @ W)


def _exact_hca(s):
    B, T, H, D = s["Q"].shape
    Hkv, m = s["K_t"].shape[2], min(len(s["K_d"]), T)
    shape, kv = (B, T, H, D), (B, T, Hkv, D)
    new = lambda sh: torch.zeros(sh, dtype=torch.float64, device=s["Q"].device)
    O, lse = new(shape), new((B, H, T))
    dQ, dK, dV = new(shape), [new(kv) for _ in range(1 + len(s["K_d"]))], [new(kv) for _ in range(1 + len(s["K_d"]))]
    causal = torch.ones(T, T, dtype=torch.bool, device=O.device).triu_(1)
    for b in range(B):
        for h in range(H):
            n = h // (H // Hkv)
            leaf = lambda x, i: x[b, :, i].double().requires_grad_(s["bwd"])
            Q, K, V = leaf(s["Q"], h), [leaf(x, n) for x in (s["K_t"], *s["K_d"])], [leaf(x, n) for x in (s["V_t"], *s["V_d"])]
            S = Q @ K[0].T
            for i in range(m):
                S = S.diagonal_scatter((Q[i:] * K[1 + i][:T - i]).sum(1), -i)
            S = (S * D ** -0.5).masked_fill(causal, -math.inf)
            P = S.softmax(1)
            near = torch.ones_like(causal).triu_(-(m - 1)) if m else torch.zeros_like(causal)
            o = P.masked_fill(near, 0.0) @ V[0]
            for i in range(m):
                o = o + torch.nn.functional.pad(P.diagonal(-i)[:, None] * V[1 + i][:T - i], (0, 0, i, 0))
            O[b, :, h], lse[b, h] = o.detach(), S.detach().logsumexp(1)
            if s["bwd"]:
                grads = torch.autograd.grad(o, [Q, *K, *V], s["dO"][b, :, h].double(), allow_unused=True)
                dQ[b, :, h] = grads[0]
                for x, gx in zip(dK + dV, grads[1:]):
                    if gx is not None:
                        x[b, :, n] += gx
    out = {"O": O, "lse": lse}
    if s["bwd"]:
        out.update(dQ=dQ, dK_t=dK[0], dV_t=dV[0], dK_d=dK[1:], dV_d=dV[1:])
    return out
