// The calls of the binding that a training step makes, from Python objects to the C entry point in native code: checks,
// output tensors, pointers. Each takes the arguments of the Python function of its name as positions (tensors, or None where that takes
// None; the stream's handle or None) and returns
//   a dict            the outputs
//   an int            the C entry point's status, where it is not HASS_OK
//   None              anything that is not the plain case: the Python function does the call itself, with its own checks and errors.
// Short calls were bound by the binding in Python (checks, eleven output tensors, ctypes; us per pass among others, before -> after): attention
// of 2 x 333 positions, 4 / 2 heads, forward + backward 55.0 -> 42.8, of 5 x 48, 2 / 1 heads 49.1 -> 25.2, forward of 2 x 86, 32 / 8 heads
// 18.5 -> 11.0; 64 rows x 256 x 1024 25.9 -> 22.1, a row alone 26.0 -> 17.3. First passes gain as much (alone: 93 -> 60, 52 -> 41).
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cmath>
#include <cstdint>
#include <vector>

#include "../../include/hass.h"

namespace {

// The library's entry points, as the binding has loaded them
struct Entries {
    decltype(&hass_topk_distill_fwd) fwd;
    decltype(&hass_topk_distill_fwd_draft) fwd_draft;
    decltype(&hass_topk_distill_bwd) bwd;
    decltype(&hass_topk_distill_fwd_bwd) fwd_bwd;
    decltype(&hass_topk_distill_fwd_bwd_draft) fwd_bwd_draft;
    decltype(&hass_combined_distill_fwd_bwd) combined;
    decltype(&hass_variant_distill_fwd_bwd) variant;
    decltype(&hass_hca_attention_fwd) hca_fwd;
    decltype(&hass_hca_attention_bwd) hca_bwd;
} lib;

const at::Tensor* tensor(PyObject* o) { return THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr; }

// A contiguous CUDA tensor of this type, or nothing
const at::Tensor* plain(PyObject* o, at::ScalarType type) {
    const at::Tensor* t = tensor(o);
    return t && t->scalar_type() == type && t->is_cuda() && t->is_contiguous() ? t : nullptr;
}

bool integer(PyObject* o, int64_t& v) {
    if (!PyLong_CheckExact(o)) return false;
    v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) {
        PyErr_Clear();
        return false;
    }
    return v >= INT32_MIN && v <= INT32_MAX;
}
bool number(PyObject* o, float& v) {
    if (!PyFloat_CheckExact(o)) return false;
    v = static_cast<float>(PyFloat_AS_DOUBLE(o));
    return true;
}

at::Tensor make(at::IntArrayRef size, at::ScalarType type, const at::Tensor& like) {
    return at::empty(size, at::TensorOptions().dtype(type).device(like.device()));
}

struct Dict {
    PyObject* d = PyDict_New();
    void put(const char* key, PyObject* v) {
        if (v) PyDict_SetItemString(d, key, v);
        Py_XDECREF(v);
    }
    void put(const char* key, const at::Tensor& t) { put(key, THPVariable_Wrap(t)); }
};

struct Call {
    const at::Tensor* ws = nullptr;
    void* stream = nullptr;
    // workspace and stream: the last two arguments of every call
    bool take(PyObject* workspace, PyObject* strm) {
        ws = plain(workspace, at::kByte);
        if (!ws) return false;
        if (strm == Py_None) {
            stream = c10::cuda::getCurrentCUDAStream().stream();
            return true;
        }
        stream = PyLong_AsVoidPtr(strm);
        if (stream == nullptr && PyErr_Occurred()) {
            PyErr_Clear();
            return false;
        }
        return true;
    }
    template <typename F, typename... A>
    int run(F f, A... a) const {
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = f(a..., ws->data_ptr(), static_cast<size_t>(ws->numel()), stream);
        Py_END_ALLOW_THREADS
        return rc;
    }
};

// H [N, d] and W [V, d]
struct Head {
    const at::Tensor *H_t = nullptr, *H_d = nullptr, *W = nullptr;
    int64_t N = 0, d = 0, V = 0, K = 0;
    bool take(PyObject* ht, PyObject* hd, PyObject* w) {
        H_d = plain(hd, at::kBFloat16);
        W = plain(w, at::kBFloat16);
        if (!H_d || !W || H_d->dim() != 2 || W->dim() != 2 || H_d->size(1) != W->size(1)) return false;
        N = H_d->size(0), d = H_d->size(1), V = W->size(0);
        if (ht) {
            H_t = plain(ht, at::kBFloat16);
            if (!H_t || H_t->sizes() != H_d->sizes()) return false;
        }
        return true;
    }
    bool rows(PyObject* o, const float*& p) const {      // fp32 [N] or None (autograd's gradient of a sum is an expanded element: not the plain case)
        p = nullptr;
        if (o == Py_None) return true;
        const at::Tensor* t = plain(o, at::kFloat);
        if (!t || t->dim() != 1 || t->size(0) != N) return false;
        p = static_cast<const float*>(t->data_ptr());
        return true;
    }
    bool set(PyObject* idx, PyObject* q, const int32_t*& pi, const float*& pq) {
        const at::Tensor *i = plain(idx, at::kInt), *v = plain(q, at::kFloat);
        if (!i || !v || i->dim() != 2 || i->size(0) != N || i->sizes() != v->sizes()) return false;
        K = i->size(1);
        if (K > INT32_MAX) return false;
        pi = static_cast<const int32_t*>(i->data_ptr());
        pq = static_cast<const float*>(v->data_ptr());
        return true;
    }
};

bool type_of(PyObject* o, int& code, at::ScalarType& type) {
    int64_t c;
    if (!integer(o, c) || (c != HASS_BF16 && c != HASS_FP32)) return false;
    code = static_cast<int>(c);
    type = c == HASS_FP32 ? at::kFloat : at::kBFloat16;
    return true;
}

#define F32(t) static_cast<float*>((t).data_ptr())
#define I32(t) static_cast<int32_t*>((t).data_ptr())
#define DEFER Py_RETURN_NONE
#define ENTRY(name, count)                                                        \
    PyObject* name##_(PyObject* const* a);                                        \
    PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n) {                 \
        if (n != count) DEFER;                                                    \
        HANDLE_TH_ERRORS                                                          \
        return name##_(a);                                                        \
        END_HANDLE_TH_ERRORS                                                      \
    }                                                                             \
    PyObject* name##_(PyObject* const* a)

// H_t, H_d, W, K, workspace, stream
ENTRY(topk_distill_fwd, 6) {
    Head h;
    Call c;
    if (!h.take(a[0], a[1], a[2]) || !integer(a[3], h.K) || h.K < 1 || !c.take(a[4], a[5])) DEFER;
    const at::Tensor loss = make({h.N}, at::kFloat, *h.H_t), idx = make({h.N, h.K}, at::kInt, *h.H_t), q = make({h.N, h.K}, at::kFloat, *h.H_t),
                     lse_t = make({h.N}, at::kFloat, *h.H_t), lse_d = make({h.N}, at::kFloat, *h.H_t);
    const int rc = c.run(lib.fwd, h.H_t->data_ptr(), h.H_d->data_ptr(), h.W->data_ptr(), h.N, h.d, h.V, static_cast<int32_t>(h.K), F32(loss),
                         I32(idx), F32(q), F32(lse_t), F32(lse_d));
    if (rc != HASS_OK) return PyLong_FromLong(rc);
    Dict o;
    o.put("loss", loss);
    o.put("topk_idx", idx);
    o.put("topk_q", q);
    o.put("lse_t", lse_t);
    o.put("lse_d", lse_d);
    return o.d;
}

// H_d, W, topk_idx, topk_q, workspace, stream
ENTRY(topk_distill_fwd_draft, 6) {
    Head h;
    Call c;
    const int32_t* idx;
    const float* q;
    if (!h.take(nullptr, a[0], a[1]) || !h.set(a[2], a[3], idx, q) || !c.take(a[4], a[5])) DEFER;
    const at::Tensor loss = make({h.N}, at::kFloat, *h.H_d), lse_d = make({h.N}, at::kFloat, *h.H_d);
    const int rc = c.run(lib.fwd_draft, h.H_d->data_ptr(), h.W->data_ptr(), h.N, h.d, h.V, static_cast<int32_t>(h.K), idx, q, F32(loss), F32(lse_d));
    if (rc != HASS_OK) return PyLong_FromLong(rc);
    Dict o;
    o.put("loss", loss);
    o.put("lse_d", lse_d);
    return o.d;
}

// H_d, W, topk_idx, topk_q, lse_d, grad_loss, dH_dtype, workspace, stream; the dict holds dH_d alone
ENTRY(topk_distill_bwd, 9) {
    Head h;
    Call c;
    const int32_t* idx;
    const float *q, *lse = nullptr, *g;
    int code;
    at::ScalarType type;
    if (!h.take(nullptr, a[0], a[1]) || !h.set(a[2], a[3], idx, q) || a[4] == Py_None || !h.rows(a[4], lse) || !h.rows(a[5], g) ||
        !type_of(a[6], code, type) || !c.take(a[7], a[8]))
        DEFER;
    const at::Tensor dH = make({h.N, h.d}, type, *h.H_d);
    const int rc = c.run(lib.bwd, h.H_d->data_ptr(), h.W->data_ptr(), h.N, h.d, h.V, static_cast<int32_t>(h.K), idx, q, lse, g, dH.data_ptr(), code);
    if (rc != HASS_OK) return PyLong_FromLong(rc);
    Dict o;
    o.put("dH_d", dH);
    return o.d;
}

// H_t, H_d, W, K, grad_loss, dH_dtype, workspace, stream
ENTRY(topk_distill_fwd_bwd, 8) {
    Head h;
    Call c;
    const float* g;
    int code;
    at::ScalarType type;
    if (!h.take(a[0], a[1], a[2]) || !integer(a[3], h.K) || h.K < 1 || !h.rows(a[4], g) || !type_of(a[5], code, type) || !c.take(a[6], a[7])) DEFER;
    const at::Tensor loss = make({h.N}, at::kFloat, *h.H_t), idx = make({h.N, h.K}, at::kInt, *h.H_t), q = make({h.N, h.K}, at::kFloat, *h.H_t),
                     lse_t = make({h.N}, at::kFloat, *h.H_t), lse_d = make({h.N}, at::kFloat, *h.H_t), dH = make({h.N, h.d}, type, *h.H_t);
    const int rc = c.run(lib.fwd_bwd, h.H_t->data_ptr(), h.H_d->data_ptr(), h.W->data_ptr(), h.N, h.d, h.V, static_cast<int32_t>(h.K), g, F32(loss),
                         I32(idx), F32(q), F32(lse_t), F32(lse_d), dH.data_ptr(), code);
    if (rc != HASS_OK) return PyLong_FromLong(rc);
    Dict o;
    o.put("loss", loss);
    o.put("topk_idx", idx);
    o.put("topk_q", q);
    o.put("lse_t", lse_t);
    o.put("lse_d", lse_d);
    o.put("dH_d", dH);
    return o.d;
}

// H_d, W, topk_idx, topk_q, grad_loss, dH_dtype, workspace, stream
ENTRY(topk_distill_fwd_bwd_draft, 8) {
    Head h;
    Call c;
    const int32_t* idx;
    const float *q, *g;
    int code;
    at::ScalarType type;
    if (!h.take(nullptr, a[0], a[1]) || !h.set(a[2], a[3], idx, q) || !h.rows(a[4], g) || !type_of(a[5], code, type) || !c.take(a[6], a[7])) DEFER;
    const at::Tensor loss = make({h.N}, at::kFloat, *h.H_d), lse_d = make({h.N}, at::kFloat, *h.H_d), dH = make({h.N, h.d}, type, *h.H_d);
    const int rc = c.run(lib.fwd_bwd_draft, h.H_d->data_ptr(), h.W->data_ptr(), h.N, h.d, h.V, static_cast<int32_t>(h.K), idx, q, g, F32(loss),
                         F32(lse_d), dH.data_ptr(), code);
    if (rc != HASS_OK) return PyLong_FromLong(rc);
    Dict o;
    o.put("loss", loss);
    o.put("lse_d", lse_d);
    o.put("dH_d", dH);
    return o.d;
}

// H_t, H_d, W, K, w_topk, grad_loss, dH_dtype, workspace, stream
ENTRY(combined_distill_fwd_bwd, 9) {
    Head h;
    Call c;
    const float* g;
    float w;
    int code;
    at::ScalarType type;
    if (!h.take(a[0], a[1], a[2]) || !integer(a[3], h.K) || h.K < 1 || !number(a[4], w) || !h.rows(a[5], g) || !type_of(a[6], code, type) ||
        !c.take(a[7], a[8]))
        DEFER;
    const at::Tensor ce = make({h.N}, at::kFloat, *h.H_t), loss = make({h.N}, at::kFloat, *h.H_t), idx = make({h.N, h.K}, at::kInt, *h.H_t),
                     q = make({h.N, h.K}, at::kFloat, *h.H_t), lse_t = make({h.N}, at::kFloat, *h.H_t), lse_d = make({h.N}, at::kFloat, *h.H_t),
                     dH = make({h.N, h.d}, type, *h.H_t);
    const int rc = c.run(lib.combined, h.H_t->data_ptr(), h.H_d->data_ptr(), h.W->data_ptr(), h.N, h.d, h.V, static_cast<int32_t>(h.K), w, g, F32(ce),
                         F32(loss), I32(idx), F32(q), F32(lse_t), F32(lse_d), dH.data_ptr(), code);
    if (rc != HASS_OK) return PyLong_FromLong(rc);
    Dict o;
    o.put("loss_ce", ce);
    o.put("loss", loss);
    o.put("topk_idx", idx);
    o.put("topk_q", q);
    o.put("lse_t", lse_t);
    o.put("lse_d", lse_d);
    o.put("dH_d", dH);
    return o.d;
}

// H_t, H_d, W, K, variant, param, grad_loss, dH_dtype, workspace, stream
ENTRY(variant_distill_fwd_bwd, 10) {
    Head h;
    Call c;
    const float* g;
    float param;
    int code;
    int64_t variant;
    at::ScalarType type;
    if (!h.take(a[0], a[1], a[2]) || !integer(a[3], h.K) || h.K < 1 || !integer(a[4], variant) || !number(a[5], param) || !h.rows(a[6], g) ||
        !type_of(a[7], code, type) || !c.take(a[8], a[9]))
        DEFER;
    const int64_t kk = variant == HASS_LOSS_BIDIR_TOPK ? 2 * h.K : h.K;      // the bi-directional set holds up to 2K tokens
    const at::Tensor loss = make({h.N}, at::kFloat, *h.H_t), idx = make({h.N, kk}, at::kInt, *h.H_t), q = make({h.N, kk}, at::kFloat, *h.H_t),
                     n = make({h.N}, at::kInt, *h.H_t), lse_t = make({h.N}, at::kFloat, *h.H_t),
                     // (Normed Top-K leaves it out)
                     lse_d = variant == HASS_LOSS_NORMED_TOPK ? at::zeros({h.N}, at::TensorOptions().dtype(at::kFloat).device(h.H_t->device()))
                                                              : make({h.N}, at::kFloat, *h.H_t),
                     dH = make({h.N, h.d}, type, *h.H_t);
    const int rc = c.run(lib.variant, h.H_t->data_ptr(), h.H_d->data_ptr(), h.W->data_ptr(), h.N, h.d, h.V, static_cast<int32_t>(h.K),
                         static_cast<int>(variant), param, g, F32(loss), I32(idx), F32(q), I32(n), F32(lse_t), F32(lse_d), dH.data_ptr(), code);
    if (rc != HASS_OK) return PyLong_FromLong(rc);
    Dict o;
    o.put("loss", loss);
    o.put("topk_idx", idx);
    o.put("topk_q", q);
    o.put("topk_n", n);
    o.put("lse_t", lse_t);
    o.put("lse_d", lse_d);
    o.put("dH_d", dH);
    return o.d;
}

// Q [B, T, H, D]; K_t, V_t and the draft passes' [B, T, Hkv, D]
struct Attention {
    const at::Tensor *Q = nullptr, *K = nullptr, *V = nullptr;
    std::vector<const void*> K_d, V_d;
    int64_t B = 0, T = 0, H = 0, Hkv = 0, D = 0;
    float scale = 0.f;
    bool list(PyObject* o, std::vector<const void*>& to) const {
        if (!PyList_CheckExact(o) && !PyTuple_CheckExact(o)) return false;
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(o);
        for (Py_ssize_t i = 0; i < n; ++i) {
            const at::Tensor* t = plain(PySequence_Fast_GET_ITEM(o, i), at::kBFloat16);
            if (!t || t->sizes() != K->sizes()) return false;
            to.push_back(t->data_ptr());
        }
        return true;
    }
    bool take(PyObject* q, PyObject* k, PyObject* v, PyObject* kd, PyObject* vd, PyObject* sc) {
        Q = plain(q, at::kBFloat16);
        K = plain(k, at::kBFloat16);
        V = plain(v, at::kBFloat16);
        if (!Q || !K || !V || Q->dim() != 4 || K->dim() != 4) return false;
        B = Q->size(0), T = Q->size(1), H = Q->size(2), D = Q->size(3), Hkv = K->size(2);
        if (K->size(0) != B || K->size(1) != T || K->size(3) != D || V->sizes() != K->sizes()) return false;
        if (!list(kd, K_d) || !list(vd, V_d) || K_d.size() != V_d.size()) return false;
        if (sc == Py_None) {
            scale = static_cast<float>(1.0 / std::sqrt(static_cast<double>(D)));
            return true;
        }
        return number(sc, scale);
    }
    int32_t m() const { return static_cast<int32_t>(K_d.size()); }
};

PyObject* tensor_list(const std::vector<at::Tensor>& v) {
    PyObject* l = PyList_New(static_cast<Py_ssize_t>(v.size()));
    for (size_t i = 0; l && i < v.size(); ++i) PyList_SET_ITEM(l, static_cast<Py_ssize_t>(i), THPVariable_Wrap(v[i]));
    return l;
}

// Q, K_t, V_t, K_d, V_d, scale, want_lse, workspace, stream
ENTRY(hca_attention_fwd, 9) {
    Attention t;
    Call c;
    if (!t.take(a[0], a[1], a[2], a[3], a[4], a[5]) || !PyBool_Check(a[6]) || !c.take(a[7], a[8])) DEFER;
    const at::Tensor O = make(t.Q->sizes(), at::kBFloat16, *t.Q);
    at::Tensor lse;
    if (a[6] == Py_True) lse = make({t.B, t.H, t.T}, at::kFloat, *t.Q);
    const int rc = c.run(lib.hca_fwd, t.Q->data_ptr(), t.K->data_ptr(), t.V->data_ptr(), t.K_d.data(), t.V_d.data(), t.m(), t.B, t.T, t.H, t.Hkv, t.D,
                         t.scale, O.data_ptr(), lse.defined() ? F32(lse) : nullptr);
    if (rc != HASS_OK) return PyLong_FromLong(rc);
    Dict o;
    o.put("O", O);
    o.put("lse", lse);      // (None where it is undefined)
    return o.d;
}

// Q, K_t, V_t, K_d, V_d, O, lse, dO, scale, workspace, stream
ENTRY(hca_attention_bwd, 11) {
    Attention t;
    Call c;
    if (!t.take(a[0], a[1], a[2], a[3], a[4], a[8]) || !c.take(a[9], a[10])) DEFER;
    const at::Tensor *O = plain(a[5], at::kBFloat16), *lse = plain(a[6], at::kFloat), *dO = plain(a[7], at::kBFloat16);
    if (!O || !lse || !dO || O->sizes() != t.Q->sizes() || dO->sizes() != t.Q->sizes() || lse->dim() != 3 || lse->size(0) != t.B ||
        lse->size(1) != t.H || lse->size(2) != t.T)
        DEFER;
    const at::Tensor dQ = make(t.Q->sizes(), at::kBFloat16, *t.Q), dK = make(t.K->sizes(), at::kBFloat16, *t.Q),
                     dV = make(t.K->sizes(), at::kBFloat16, *t.Q);
    std::vector<at::Tensor> dK_d, dV_d;
    std::vector<void*> pk, pv;
    for (int i = 0; i < t.m(); ++i) {
        dK_d.push_back(make(t.K->sizes(), at::kBFloat16, *t.Q));
        dV_d.push_back(make(t.K->sizes(), at::kBFloat16, *t.Q));
        pk.push_back(dK_d.back().data_ptr());
        pv.push_back(dV_d.back().data_ptr());
    }
    const int rc = c.run(lib.hca_bwd, t.Q->data_ptr(), t.K->data_ptr(), t.V->data_ptr(), t.K_d.data(), t.V_d.data(), t.m(), t.B, t.T, t.H, t.Hkv, t.D,
                         t.scale, O->data_ptr(), static_cast<const float*>(lse->data_ptr()), dO->data_ptr(), dQ.data_ptr(), dK.data_ptr(),
                         dV.data_ptr(), pk.data(), pv.data());
    if (rc != HASS_OK) return PyLong_FromLong(rc);
    Dict o;
    o.put("dQ", dQ);
    o.put("dK_t", dK);
    o.put("dV_t", dV);
    o.put("dK_d", tensor_list(dK_d));
    o.put("dV_d", tensor_list(dV_d));
    return o.d;
}

// The addresses of the library's entry points, in the order of Entries
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    void** to = reinterpret_cast<void**>(&lib);
    if (n != static_cast<Py_ssize_t>(sizeof(lib) / sizeof(void*))) {
        PyErr_SetString(PyExc_ValueError, "bind: one address per entry point");
        return nullptr;
    }
    for (Py_ssize_t i = 0; i < n; ++i) {
        to[i] = PyLong_AsVoidPtr(a[i]);
        if (to[i] == nullptr) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "bind: a null address");
            return nullptr;
        }
    }
    Py_RETURN_NONE;
}

#define METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(bind), METHOD(topk_distill_fwd), METHOD(topk_distill_fwd_draft), METHOD(topk_distill_bwd), METHOD(topk_distill_fwd_bwd),
                         METHOD(topk_distill_fwd_bwd_draft), METHOD(combined_distill_fwd_bwd), METHOD(variant_distill_fwd_bwd),
                         METHOD(hca_attention_fwd), METHOD(hca_attention_bwd), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "hass_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_hass_host(void) { return PyModule_Create(&module); }
