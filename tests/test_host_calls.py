"""The native form of the binding's calls: the same outputs as the Python form, which does everything that is not the plain case."""
import os
import sysconfig

import pytest
import torch

import paper_2408_15766_b200 as hass
from paper_2408_15766_b200 import binding


class _Nothing:
    """Every native call defers."""

    def __getattr__(self, name):
        return lambda *args: None


def _tensors(v):
    for x in v if isinstance(v, (list, tuple)) else [v]:
        yield x


@pytest.mark.gpu
@pytest.mark.parametrize("grad", [False, True])
def test_native_and_python_forms_agree(monkeypatch, grad):
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(3)
    R = lambda *s: torch.randn(*s, generator=g, device=dev).to(torch.bfloat16)
    N, d, V, K = 37, 128, 1500, 7
    H_t, H_d, W = R(N, d), R(N, d), R(V, d)
    gl = torch.rand(N, generator=g, device=dev) if grad else None
    ws = torch.empty(hass.combined_distill_workspace_bytes(N, d, V, K), dtype=torch.uint8, device=dev)
    f = hass.topk_distill_fwd(H_t, H_d, W, K, workspace=ws)
    B, T, H, Hkv, m = 2, 150, 4, 2, 2 if grad else 0
    Q, Kt, Vt, dO = R(B, T, H, 128), R(B, T, Hkv, 128), R(B, T, Hkv, 128), R(B, T, H, 128)
    Kd, Vd = [R(B, T, Hkv, 128) for _ in range(m)], tuple(R(B, T, Hkv, 128) for _ in range(m))
    wa = torch.empty(hass.hca_attention_workspace_bytes(), dtype=torch.uint8, device=dev)
    wb = torch.empty(hass.hca_attention_bwd_workspace_bytes(B, T, H, m), dtype=torch.uint8, device=dev)
    scale = 0.1 if grad else None
    stream = torch.cuda.current_stream() if grad else None
    fw = hass.hca_attention_fwd(Q, Kt, Vt, Kd, Vd, scale, workspace=wa)
    dtype = hass.HASS_FP32 if grad else hass.HASS_BF16
    calls = {
        "fwd": lambda: hass.topk_distill_fwd(H_t, H_d, W, K, workspace=ws, stream=stream),
        "fwd_draft": lambda: hass.topk_distill_fwd_draft(H_d, W, f["topk_idx"], f["topk_q"], workspace=ws, stream=stream),
        "bwd": lambda: {"dH": hass.topk_distill_bwd(H_d, W, f["topk_idx"], f["topk_q"], f["lse_d"], gl, dtype, workspace=ws, stream=stream)},
        "fwd_bwd": lambda: hass.topk_distill_fwd_bwd(H_t, H_d, W, K, gl, dtype, workspace=ws, stream=stream),
        "fwd_bwd_draft": lambda: hass.topk_distill_fwd_bwd_draft(H_d, W, f["topk_idx"], f["topk_q"], gl, dtype, workspace=ws),
        "combined": lambda: hass.combined_distill_fwd_bwd(H_t, H_d, W, K, 0.5, gl, dtype, workspace=ws),
        "top_p": lambda: hass.variant_distill_fwd_bwd(H_t, H_d, W, K, hass.LOSS_TOP_P, 0.01, gl, dtype, workspace=ws),
        "normed": lambda: hass.variant_distill_fwd_bwd(H_t, H_d, W, K, hass.LOSS_NORMED_TOPK, grad_loss=gl, dH_dtype=dtype, workspace=ws),
        "bidir": lambda: hass.variant_distill_fwd_bwd(H_t, H_d, W, K, hass.LOSS_BIDIR_TOPK, grad_loss=gl, dH_dtype=dtype, workspace=ws),
        "hca_fwd": lambda: hass.hca_attention_fwd(Q, Kt, Vt, Kd, Vd, scale, not grad, workspace=wa, stream=stream),
        "hca_bwd": lambda: hass.hca_attention_bwd(Q, Kt, Vt, Kd, Vd, fw["O"], fw["lse"], dO, scale, workspace=wb, stream=stream),
    }
    native = {name: call() for name, call in calls.items()}
    monkeypatch.setattr(binding, "_host", _Nothing())
    for name, call in calls.items():
        a, b = native[name], call()
        assert list(a) == list(b), name
        for key in b:
            if key == "workspace":
                assert a[key] is b[key]
                continue
            for x, y in zip(_tensors(a[key]), _tensors(b[key]), strict=True):
                assert (x is None) == (y is None), (name, key)
                if x is not None:
                    assert x.dtype == y.dtype and x.shape == y.shape and x.is_contiguous() and not x.requires_grad, (name, key)
                    # (dQ is a sum in no fixed order, rounded to bf16)
                    assert torch.equal(x, y) if key != "dQ" else torch.allclose(x.float(), y.float(), rtol=2.0 ** -7, atol=1e-3), (name, key)


# What autograd hands a per-row loss: behind .sum() one element for all rows, behind an indexed sum every second of a longer buffer. (Both lie in
# buffers that N floats from their first element on do not leave.)
@pytest.mark.gpu
@pytest.mark.parametrize("native", [True, False])
@pytest.mark.parametrize("layout", ["expanded", "strided"])
def test_grad_loss_of_any_stride(monkeypatch, native, layout):
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(4)
    R = lambda *s: torch.randn(*s, generator=g, device=dev).to(torch.bfloat16)
    N, d, V, K = 37, 128, 1500, 7
    H_t, H_d, W = R(N, d), R(N, d), R(V, d)
    buf = torch.rand(2 * N, generator=g, device=dev)
    gl = (buf[:1].expand(N) if layout == "expanded" else buf[::2]).requires_grad_()
    plain = torch.tensor(gl.tolist(), device=dev)
    ws = torch.empty(hass.combined_distill_workspace_bytes(N, d, V, K), dtype=torch.uint8, device=dev)
    f = hass.topk_distill_fwd(H_t, H_d, W, K, workspace=ws)
    host = {k: v.cpu() for k, v in {"H_t": H_t, "H_d": H_d}.items()}

    def from_host(w):
        loss, dH = torch.empty(N), torch.empty(N, d, dtype=torch.bfloat16)
        hass.topk_distill_fwd_bwd_host(host["H_t"], host["H_d"], W, K, loss, dH, w.cpu() if w is plain else w.detach().cpu().as_strided((N,), (0,)) if
                                       layout == "expanded" else buf.cpu()[::2])
        return dH

    if not native:
        monkeypatch.setattr(binding, "_host", _Nothing())
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    calls = {
        "bwd": lambda w: hass.topk_distill_bwd(H_d, W, f["topk_idx"], f["topk_q"], f["lse_d"], w, workspace=ws),
        "fwd_bwd": lambda w: hass.topk_distill_fwd_bwd(H_t, H_d, W, K, w, workspace=ws)["dH_d"],
        "fwd_bwd_draft": lambda w: hass.topk_distill_fwd_bwd_draft(H_d, W, f["topk_idx"], f["topk_q"], w, workspace=ws)["dH_d"],
        "combined": lambda w: hass.combined_distill_fwd_bwd(H_t, H_d, W, K, 0.5, w, workspace=ws)["dH_d"],
        "normed": lambda w: hass.variant_distill_fwd_bwd(H_t, H_d, W, K, hass.LOSS_NORMED_TOPK, grad_loss=w, workspace=ws)["dH_d"],
        "bidir": lambda w: hass.variant_distill_fwd_bwd(H_t, H_d, W, K, hass.LOSS_BIDIR_TOPK, grad_loss=w, workspace=ws)["dH_d"],
        "host": from_host,
        "side": lambda w: hass.topk_distill_fwd_bwd(H_t, H_d, W, K, w, workspace=ws, stream=side)["dH_d"],
    }
    for name, call in calls.items():
        a, b = call(gl), call(plain)
        torch.cuda.synchronize()
        assert torch.equal(a, b) and not a.requires_grad, name
        if name != "host":
            assert torch.equal(call(plain.cpu()), b), name      # (pageable memory: a copy on the GPU)


@pytest.mark.gpu
def test_a_status_is_the_same_error_in_both_forms(monkeypatch):
    dev = torch.device("cuda:0")
    x = torch.zeros(4, 64, dtype=torch.bfloat16, device=dev)
    ws = torch.empty(256, dtype=torch.uint8, device=dev)
    for host in (binding._host, _Nothing()):
        monkeypatch.setattr(binding, "_host", host)
        with pytest.raises(hass.HassError) as e:
            hass.topk_distill_fwd_bwd(x, x, x, 2, workspace=ws)
        assert e.value.status == -3
        with pytest.raises(hass.HassError) as e:
            hass.topk_distill_fwd(x, x, x, 65, workspace=ws)
        assert e.value.status == -1


def test_what_is_not_the_plain_case_is_left_to_python():
    x = torch.zeros(4, 64, dtype=torch.bfloat16)
    ws = torch.empty(1 << 16, dtype=torch.uint8)
    assert binding._host.topk_distill_fwd_bwd(x, x, x, 2, None, 0, ws, None) is None          # no CUDA tensors
    assert binding._host.topk_distill_fwd(x, x, x, 2, None, None) is None                     # no workspace
    assert binding._host.topk_distill_fwd(x, x, "W", 2, ws, None) is None
    assert binding._host.hca_attention_fwd(x, x, x, [], [], None, True, ws, None) is None
    assert binding._host.topk_distill_fwd(x) is None
    with pytest.raises(AssertionError):
        hass.topk_distill_fwd_bwd(x, x, x.float(), 2)
    with pytest.raises(AssertionError):
        hass.topk_distill_fwd_bwd(x, x, x, 2, workspace=ws)


def test_native_calls_of_another_torch_are_not_loaded(tmp_path):
    """Their file is named after torch and Python; where it is missing the package loads and every call is left to its Python form."""
    name = os.path.basename(binding.HOST)
    assert torch.__version__ in name and name.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    assert binding._host.__file__ == binding.HOST
    with pytest.warns(UserWarning, match="is missing"):
        host = binding._load_host(binding.lib, str(tmp_path / "hass_host-0.0.so"))
    x = torch.zeros(4, 64, dtype=torch.bfloat16)
    assert host.topk_distill_fwd(x, x, x, 2, None, None) is None
