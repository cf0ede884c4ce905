// Argument marshalling of the Python binding in native code: reads the tensors' pointers, sizes and strides,
// allocates what the call returns, fills a psk_shape and calls the C ABI (whose entry points binding.py
// hands over as addresses, so that both use the same library).  A call through ctypes spends 15-40 us in
// Python on this, more than the kernels of a decode step or of a short forward take; here it is 3-6 us.
// Every function returns None for arguments that need a closer look (not on a CUDA device, layouts
// that differ, a missing workspace ...): binding.py then checks them one by one and raises.  Otherwise the
// library's status (an int) if it is not 0, or the results.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <ATen/ATen.h>
#include <ATen/cuda/CUDAContextLight.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "psk.h"

namespace {

struct Api {
    decltype(&psk_workspace_bytes) workspace_bytes;
    decltype(&psk_causal_attn_fwd) attn_fwd;
    decltype(&psk_causal_attn_bwd) attn_bwd;
    decltype(&psk_lt_multiply_workspace_bytes) lt_bytes;
    decltype(&psk_lt_multiply) lt;
    decltype(&psk_lt_multiply_bf16_workspace_bytes) lt16_bytes;
    decltype(&psk_lt_multiply_bf16) lt16;
    decltype(&psk_decode_step) decode;
    decltype(&psk_learned_workspace_bytes) learned_bytes;
    decltype(&psk_learned_attn_fwd) learned_fwd;
    decltype(&psk_learned_attn_bwd) learned_bwd;
} api;

using at::Tensor;

// A tensor argument, nullptr for None; `ok` becomes false for anything else.
const Tensor* tensor(PyObject* o, bool& ok) {
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) { ok = false; return nullptr; }
    return &THPVariable_Unpack(o);
}
const Tensor* cuda_tensor(PyObject* o, bool& ok) {
    const Tensor* t = tensor(o, ok);
    if (t == nullptr || !t->is_cuda()) ok = false;
    return t;
}
int integer(PyObject* o, bool& ok) {
    const long v = PyLong_Check(o) ? PyLong_AsLong(o) : -1;
    if (!PyLong_Check(o) || v < INT32_MIN || v > INT32_MAX) { ok = false; PyErr_Clear(); return 0; }
    return (int)v;
}
void* ptr(const Tensor* t) { return t != nullptr ? t->data_ptr() : nullptr; }
bool same_layout(const Tensor& a, const Tensor* b) {
    return b != nullptr && b->scalar_type() == a.scalar_type() && b->sizes() == a.sizes() && b->strides() == a.strides();
}
Tensor empty_as(const Tensor& x) { return at::detail::empty_strided_cuda(x.sizes(), x.strides(), x.scalar_type(), x.device()); }
Tensor empty(at::IntArrayRef sizes, at::ScalarType type, const Tensor& like) {
    return at::detail::empty_cuda(sizes, type, like.device(), c10::nullopt);
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

bool make_shape(const Tensor& q, const Tensor* G1, int r, int b, int p, int path, int flags, int segs, psk_shape* s) {
    if (q.dim() != 4 || q.stride(3) != 1) return false;
    if (q.scalar_type() != at::kFloat && q.scalar_type() != at::kBFloat16) return false;
    for (int i = 0; i < 4; ++i) if (q.size(i) > INT32_MAX) return false;
    *s = psk_shape{(int32_t)q.size(0), (int32_t)q.size(1), (int32_t)q.size(2), (int32_t)q.size(3), r, p, b,
                   q.scalar_type() == at::kFloat ? PSK_F32 : PSK_BF16, q.stride(0), q.stride(1), q.stride(2),
                   G1 != nullptr && G1->dim() == 3 ? (int32_t)G1->size(0) : 1, path, flags, segs};
    return true;
}

// The call's scratch: the caller's, or one of the size the library asks for.
struct Scratch {
    Tensor own;
    void* p = nullptr;
    size_t n = 0;
    void take(const Tensor* given, size_t need, size_t least, const Tensor& like) {
        if (given != nullptr) { p = given->data_ptr(); n = need != 0 ? (size_t)given->numel() : 0; return; }
        if (need == 0 && least == 0) return;
        own = empty({(int64_t)(need > least ? need : least)}, at::kByte, like);
        p = own.data_ptr();
        n = need != 0 ? (size_t)own.numel() : 0;
    }
};

PyObject* status_of(int st) { return PyLong_FromLong(st); }
PyObject* tuple2(Tensor a, Tensor b) {
    PyObject* t = PyTuple_New(2);
    PyTuple_SET_ITEM(t, 0, THPVariable_Wrap(std::move(a)));
    PyTuple_SET_ITEM(t, 1, THPVariable_Wrap(std::move(b)));
    return t;
}

#define PSK_NO_GIL(st, call) do { Py_BEGIN_ALLOW_THREADS st = (call); Py_END_ALLOW_THREADS } while (0)

// (Q, K, V, G1, G2, b, p, path, workspace, out, denom, flags, seq_segments) -> (O, denom)
PyObject* attn_fwd(PyObject* const* a, Py_ssize_t n) {
    if (n != 13) Py_RETURN_NONE;
    bool ok = true;
    const Tensor *Q = cuda_tensor(a[0], ok), *K = cuda_tensor(a[1], ok), *V = cuda_tensor(a[2], ok);
    const Tensor *G1 = tensor(a[3], ok), *G2 = tensor(a[4], ok), *ws = tensor(a[8], ok), *out = tensor(a[9], ok), *den = tensor(a[10], ok);
    const int b = integer(a[5], ok), p = integer(a[6], ok), path = integer(a[7], ok), flags = integer(a[11], ok), segs = integer(a[12], ok);
    if (!ok || !same_layout(*Q, K) || !same_layout(*Q, V) || (out != nullptr && !same_layout(*Q, out))) Py_RETURN_NONE;
    if ((G1 != nullptr && (!G1->is_cuda() || !G1->is_contiguous() || G1->dim() == 0)) || (G2 != nullptr && (!G2->is_cuda() || !G2->is_contiguous()))) Py_RETURN_NONE;
    if ((flags & PSK_FLAG_KEEP_STATES) && ws == nullptr) Py_RETURN_NONE;
    psk_shape s;
    if (!make_shape(*Q, G1, 0, b, p, path, flags, segs, &s)) Py_RETURN_NONE;
    s.r = G1 != nullptr ? (int32_t)G1->size(-1) : s.h;
    Tensor O = out != nullptr ? *out : empty_as(*Q);
    Tensor d = den != nullptr ? *den : empty({s.B, s.H, s.n}, at::kFloat, *Q);
    Scratch w;
    const size_t need = api.workspace_bytes(&s, 0);
    if (need != 0) w.take(ws, need, 0, *Q);
    int st;
    void* cs = stream();
    PSK_NO_GIL(st, api.attn_fwd(&s, ptr(Q), ptr(K), ptr(V), ptr(G1), ptr(G2), O.data_ptr(), (float*)d.data_ptr(), w.p, w.n, cs));
    if (st != 0) return status_of(st);
    return tuple2(std::move(O), std::move(d));
}

// (Q, K, V, G1, G2, O, denom, dO, b, p, path, workspace, out, flags, seq_segments) -> (dQ, dK, dV)
PyObject* attn_bwd(PyObject* const* a, Py_ssize_t n) {
    if (n != 15) Py_RETURN_NONE;
    bool ok = true;
    const Tensor *Q = cuda_tensor(a[0], ok), *K = cuda_tensor(a[1], ok), *V = cuda_tensor(a[2], ok);
    const Tensor *G1 = tensor(a[3], ok), *G2 = tensor(a[4], ok), *O = cuda_tensor(a[5], ok), *den = cuda_tensor(a[6], ok), *dO = cuda_tensor(a[7], ok);
    const int b = integer(a[8], ok), p = integer(a[9], ok), path = integer(a[10], ok), flags = integer(a[13], ok), segs = integer(a[14], ok);
    const Tensor* ws = tensor(a[11], ok);
    if (!ok || !same_layout(*Q, K) || !same_layout(*Q, V) || !same_layout(*Q, O) || !same_layout(*Q, dO)) Py_RETURN_NONE;
    if ((G1 != nullptr && (!G1->is_cuda() || !G1->is_contiguous() || G1->dim() == 0)) || (G2 != nullptr && (!G2->is_cuda() || !G2->is_contiguous()))) Py_RETURN_NONE;
    if ((flags & PSK_FLAG_KEEP_STATES) && ws == nullptr) Py_RETURN_NONE;
    psk_shape s;
    if (!make_shape(*Q, G1, 0, b, p, path, flags, segs, &s)) Py_RETURN_NONE;
    s.r = G1 != nullptr ? (int32_t)G1->size(-1) : s.h;
    Tensor g[3];
    if (a[12] == Py_None) {
        for (auto& t : g) t = empty_as(*Q);
    } else {
        if (!PyTuple_Check(a[12]) || PyTuple_GET_SIZE(a[12]) != 3) Py_RETURN_NONE;
        for (int i = 0; i < 3; ++i) {
            const Tensor* t = tensor(PyTuple_GET_ITEM(a[12], i), ok);
            if (!ok || !same_layout(*Q, t)) Py_RETURN_NONE;
            g[i] = *t;
        }
    }
    Scratch w;
    const size_t need = api.workspace_bytes(&s, 1);
    if (need != 0) w.take(ws, need, 0, *Q);
    int st;
    void* cs = stream();
    PSK_NO_GIL(st, api.attn_bwd(&s, ptr(Q), ptr(K), ptr(V), ptr(G1), ptr(G2), ptr(O), (const float*)ptr(den), ptr(dO), g[0].data_ptr(),
                                g[1].data_ptr(), g[2].data_ptr(), w.p, w.n, cs));
    if (st != 0) return status_of(st);
    PyObject* t = PyTuple_New(3);
    for (int i = 0; i < 3; ++i) PyTuple_SET_ITEM(t, i, THPVariable_Wrap(std::move(g[i])));
    return t;
}

// (q, k, v, G1, G2, state) -> (o, denom)
PyObject* decode_step(PyObject* const* a, Py_ssize_t n) {
    if (n != 6) Py_RETURN_NONE;
    bool ok = true;
    const Tensor* t[6];
    for (int i = 0; i < 6; ++i) {
        t[i] = cuda_tensor(a[i], ok);
        if (!ok || !t[i]->is_contiguous()) Py_RETURN_NONE;
    }
    const Tensor &q = *t[0], &G1 = *t[3];
    if (q.dim() != 3 || G1.dim() < 2 || (q.scalar_type() != at::kFloat && q.scalar_type() != at::kBFloat16)) Py_RETURN_NONE;
    const int64_t B = q.size(0), H = q.size(1), h = q.size(2), r = G1.size(-1);
    if (B > INT32_MAX || H > INT32_MAX || h != 64 || (r != 16 && r != 32 && r != 64) || t[5]->numel() != B * H * r * r * 65) Py_RETURN_NONE;
    const psk_shape s{(int32_t)B, (int32_t)H, 1, (int32_t)h, (int32_t)r, 4, 128, q.scalar_type() == at::kFloat ? PSK_F32 : PSK_BF16, H * h, h, h,
                      G1.dim() == 3 ? (int32_t)G1.size(0) : 1, PSK_PATH_AUTO, 0, 0};
    Tensor o = at::detail::empty_cuda(q.sizes(), q.scalar_type(), q.device(), c10::nullopt), d = empty({B, H}, at::kFloat, q);
    int st;
    void* cs = stream();
    PSK_NO_GIL(st, api.decode(&s, ptr(t[0]), ptr(t[1]), ptr(t[2]), ptr(t[3]), ptr(t[4]), (float*)ptr(t[5]), o.data_ptr(), (float*)d.data_ptr(), cs));
    if (st != 0) return status_of(st);
    return tuple2(std::move(o), std::move(d));
}

// (A, B, C, b, workspace, bf16) -> Out, or for bf16 (Out, workspace)
PyObject* lt_multiply(PyObject* const* a, Py_ssize_t n) {
    if (n != 6) Py_RETURN_NONE;
    bool ok = true;
    const Tensor *A = cuda_tensor(a[0], ok), *B = cuda_tensor(a[1], ok), *C = cuda_tensor(a[2], ok), *ws = tensor(a[4], ok);
    const int b = integer(a[3], ok);
    const bool half = a[5] == Py_True;
    if (!ok) Py_RETURN_NONE;
    for (const Tensor* t : {A, B, C})
        if (t->dim() != 3 || !t->is_contiguous() || t->scalar_type() != (half ? at::kBFloat16 : at::kFloat)) Py_RETURN_NONE;
    if (B->sizes() != A->sizes() || C->size(0) != A->size(0) || C->size(1) != A->size(1)) Py_RETURN_NONE;
    for (int i = 0; i < 3; ++i) if (A->size(i) > INT32_MAX || C->size(i) > INT32_MAX) Py_RETURN_NONE;
    const int batch = (int)A->size(0), rows = (int)A->size(1), m = (int)A->size(2), k = (int)C->size(2);
    Tensor out = empty({batch, rows, k}, at::kFloat, *A);
    Scratch w;
    int st;
    void* cs = stream();
    if (half) {
        w.take(ws, api.lt16_bytes(batch, rows, m, k, b), 256, *A);
        PSK_NO_GIL(st, api.lt16(batch, rows, m, k, b, ptr(A), ptr(B), ptr(C), (float*)out.data_ptr(), w.p, w.n, cs));
        if (st != 0) return status_of(st);
        return tuple2(std::move(out), ws != nullptr ? *ws : w.own);
    }
    const size_t need = api.lt_bytes(batch, rows, m, k, b);
    w.take(ws, need, 0, *A);
    if (ws != nullptr) w.n = (size_t)ws->numel();
    PSK_NO_GIL(st, api.lt(batch, rows, m, k, b, (const float*)ptr(A), (const float*)ptr(B), (const float*)ptr(C), (float*)out.data_ptr(), w.p, w.n, cs));
    if (st != 0) return status_of(st);
    return THPVariable_Wrap(std::move(out));
}

// (Q, K, V, params, r, b, flags, workspace, path) -> (O, denom)
PyObject* learned_fwd(PyObject* const* a, Py_ssize_t n) {
    if (n != 9) Py_RETURN_NONE;
    bool ok = true;
    const Tensor *Q = cuda_tensor(a[0], ok), *K = cuda_tensor(a[1], ok), *V = cuda_tensor(a[2], ok), *P = cuda_tensor(a[3], ok), *ws = tensor(a[7], ok);
    const int r = integer(a[4], ok), b = integer(a[5], ok), flags = integer(a[6], ok), path = integer(a[8], ok);
    psk_shape s;
    if (!ok || !same_layout(*Q, K) || !same_layout(*Q, V) || !make_shape(*Q, nullptr, r, b, 4, path, flags, 0, &s)) Py_RETURN_NONE;
    Scratch w;
    w.take(ws, api.learned_bytes(&s, 0), 256, *Q);
    Tensor O = empty_as(*Q), d = empty({s.B, s.H, s.n}, at::kFloat, *Q);
    int st;
    void* cs = stream();
    PSK_NO_GIL(st, api.learned_fwd(&s, ptr(Q), ptr(K), ptr(V), (const float*)ptr(P), O.data_ptr(), (float*)d.data_ptr(), w.p, w.n, cs));
    if (st != 0) return status_of(st);
    return tuple2(std::move(O), std::move(d));
}

// (Q, K, V, params, O, denom, dO, r, b, flags, workspace, path) -> (dQ, dK, dV, dparams)
PyObject* learned_bwd(PyObject* const* a, Py_ssize_t n) {
    if (n != 12) Py_RETURN_NONE;
    bool ok = true;
    const Tensor *Q = cuda_tensor(a[0], ok), *K = cuda_tensor(a[1], ok), *V = cuda_tensor(a[2], ok), *P = cuda_tensor(a[3], ok);
    const Tensor *O = cuda_tensor(a[4], ok), *den = cuda_tensor(a[5], ok), *dO = cuda_tensor(a[6], ok), *ws = tensor(a[10], ok);
    const int r = integer(a[7], ok), b = integer(a[8], ok), flags = integer(a[9], ok), path = integer(a[11], ok);
    psk_shape s;
    if (!ok || !same_layout(*Q, K) || !same_layout(*Q, V) || !same_layout(*Q, O) || !same_layout(*Q, dO) || !P->is_contiguous() ||
        !make_shape(*Q, nullptr, r, b, 4, path, flags, 0, &s)) Py_RETURN_NONE;
    Scratch w;
    w.take(ws, api.learned_bytes(&s, 1), 256, *Q);
    Tensor g[4] = {empty_as(*Q), empty_as(*Q), empty_as(*Q), empty_as(*P)};
    int st;
    void* cs = stream();
    PSK_NO_GIL(st, api.learned_bwd(&s, ptr(Q), ptr(K), ptr(V), (const float*)ptr(P), ptr(O), (const float*)ptr(den), ptr(dO), g[0].data_ptr(),
                                   g[1].data_ptr(), g[2].data_ptr(), (float*)g[3].data_ptr(), w.p, w.n, cs));
    if (st != 0) return status_of(st);
    PyObject* t = PyTuple_New(4);
    for (int i = 0; i < 4; ++i) PyTuple_SET_ITEM(t, i, THPVariable_Wrap(std::move(g[i])));
    return t;
}

// init(addresses): the C ABI's entry points in the order of `Api`.
PyObject* init(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != (Py_ssize_t)(sizeof(Api) / sizeof(void*))) { PyErr_SetString(PyExc_ValueError, "wrong number of entry points"); return nullptr; }
    void** slot = reinterpret_cast<void**>(&api);
    for (Py_ssize_t i = 0; i < n; ++i) {
        slot[i] = PyLong_AsVoidPtr(a[i]);
        if (slot[i] == nullptr) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null entry point"); return nullptr; }
    }
    Py_RETURN_NONE;
}

// C++ exceptions (out of memory among them) as torch's own Python exceptions
template <PyObject* (*F)(PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    return F(a, n);
    END_HANDLE_TH_ERRORS
}

#define PSK_M(f) {#f, (PyCFunction)(void (*)(void))guarded<f>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {{"init", (PyCFunction)(void (*)(void))init, METH_FASTCALL, nullptr}, PSK_M(attn_fwd), PSK_M(attn_bwd), PSK_M(decode_step), PSK_M(lt_multiply),
                         PSK_M(learned_fwd), PSK_M(learned_bwd), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_psk_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// BUILT_FOR: the Python and torch of the build, which binding.py compares with the running ones.
PyMODINIT_FUNC PyInit__psk_native(void) {
    PyObject* m = PyModule_Create(&module);
    if (m != nullptr && PyModule_AddStringConstant(m, "BUILT_FOR", PSK_BUILT_FOR) != 0) { Py_DECREF(m); return nullptr; }
    return m;
}
