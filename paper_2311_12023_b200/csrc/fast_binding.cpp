// Marshalling of the layer calls and of the encoder in native code.  binding.py tries these first; they answer None for everything out of the
// ordinary (tensor subclasses, wrapped tensors, wrong shapes or types, fields that are not integers), and the Python code then takes the call
// and raises what it always raised.  It takes every call where this module is missing or was compiled for another torch or Python (`built_for`,
// see build.py).  Nothing is kept between calls: every argument is looked at each time.
//
// What bounded a small call was this work in Python: linear_fwd on one row of a 4096 x 4096 matrix, host time per call 11.9 us, now 6.7, of which 5.6 are the two launches; encoder 22.6 and 9.4.
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/DispatchKeySet.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>

#include <climits>

#include "../../include/lqlora.h"

namespace {

using LinearFn = int (*)(const lqlora_qmatrix*, const void*, const void*, int, const void*, int64_t, void*, void*, size_t, void*);
using SizesFn = int (*)(int64_t, int64_t, const lqlora_config*, size_t*, size_t*, size_t*, size_t*);
using EncodeFn = int (*)(const float*, lqlora_qmatrix*, void*, size_t, void*);

LinearFn g_linear[2];
SizesFn g_sizes;
EncodeFn g_encode;
PyObject *g_parameter, *g_qmatrix;                              // torch.nn.Parameter, binding.QMatrix
PyObject *s_codes, *s_scale_codes, *s_scale2, *s_N, *s_K, *s_cfg, *s_b0, *s_B0, *s_b1, *s_B1, *s_b2;

// A dense CUDA tensor that nothing stands in front of (no subclass, no transform, no mode that keeps its storage elsewhere).
bool plain(const at::Tensor& t) {
    static const c10::DispatchKeySet allowed({c10::DispatchKey::CUDA, c10::DispatchKey::AutogradCUDA, c10::DispatchKey::ADInplaceOrView, c10::DispatchKey::AutocastCUDA});
    return t.defined() && (t.key_set() | allowed) == allowed && t.has_storage();
}
const at::Tensor* plain_tensor(PyObject* o) {
    const PyTypeObject* type = Py_TYPE(o);
    if (reinterpret_cast<PyObject*>(const_cast<PyTypeObject*>(type)) != THPVariableClass && reinterpret_cast<PyObject*>(const_cast<PyTypeObject*>(type)) != g_parameter) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    return plain(t) ? &t : nullptr;
}

// A mode that wants to see the tensor operations of a call.
bool modes() { return at::impl::torch_function_mode_enabled() || c10::impl::dispatch_mode_enabled(); }

// An integer attribute; false (no exception left) for anything else.
bool int_attr(PyObject* o, PyObject* name, int64_t lo, int64_t hi, int64_t* out) {
    PyObject* v = PyObject_GetAttr(o, name);
    if (!v) { PyErr_Clear(); return false; }
    bool ok = PyLong_Check(v);
    if (ok) {
        int overflow = 0;
        const long long x = PyLong_AsLongLongAndOverflow(v, &overflow);
        ok = overflow == 0 && x >= lo && x <= hi;
        *out = x;
    }
    Py_DECREF(v);
    return ok;
}
bool config_of(PyObject* cfg, lqlora_config* c) {
    int64_t v[5];
    PyObject* const names[5] = {s_b0, s_B0, s_b1, s_B1, s_b2};
    for (int i = 0; i < 5; ++i)
        if (!int_attr(cfg, names[i], INT_MIN, INT_MAX, &v[i])) return false;
    c->b0 = static_cast<int>(v[0]); c->B0 = static_cast<int>(v[1]); c->b1 = static_cast<int>(v[2]); c->B1 = static_cast<int>(v[3]); c->b2 = static_cast<int>(v[4]);
    return true;
}
// The address of a tensor attribute; the tensor is kept by its owner for the length of the call.
bool data_attr(PyObject* o, PyObject* name, void** out) {
    PyObject* v = PyObject_GetAttr(o, name);
    if (!v) { PyErr_Clear(); return false; }
    const at::Tensor* t = plain_tensor(v);
    if (t) *out = t->data_ptr();
    Py_DECREF(v);
    return t != nullptr;
}

// linear(backward, q, L1, L2, A, out, workspace) -> result tensor, status number of a call that failed, or None.
PyObject* linear(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 7 || !g_qmatrix || modes()) Py_RETURN_NONE;
    const bool backward = args[0] == Py_True;
    PyObject *q = args[1], *oL1 = args[2], *oL2 = args[3], *oA = args[4], *oout = args[5], *ows = args[6];
    if (reinterpret_cast<PyObject*>(Py_TYPE(q)) != g_qmatrix || reinterpret_cast<PyObject*>(Py_TYPE(oA)) != THPVariableClass) Py_RETURN_NONE;
    const at::Tensor* A = plain_tensor(oA);
    const at::Tensor* ws = plain_tensor(ows);
    if (!A || !ws || A->scalar_type() != at::kBFloat16 || A->dim() != 2 || !A->is_contiguous()) Py_RETURN_NONE;

    lqlora_qmatrix m{};
    void *codes, *sc, *s2;
    if (!data_attr(q, s_codes, &codes) || !data_attr(q, s_scale_codes, &sc) || !data_attr(q, s_scale2, &s2)) Py_RETURN_NONE;
    m.codes = codes; m.scale_codes = static_cast<uint8_t*>(sc); m.scale2 = static_cast<float*>(s2);
    int64_t N, K;
    if (!int_attr(q, s_N, 0, INT64_MAX, &N) || !int_attr(q, s_K, 0, INT64_MAX, &K)) Py_RETURN_NONE;
    m.N = N; m.K = K;
    PyObject* cfg = PyObject_GetAttr(q, s_cfg);
    if (!cfg) { PyErr_Clear(); Py_RETURN_NONE; }
    const bool cfg_ok = config_of(cfg, &m.cfg);
    Py_DECREF(cfg);
    if (!cfg_ok || A->size(1) != (backward ? N : K)) Py_RETURN_NONE;

    int r = 0;
    const void *L1p = nullptr, *L2p = nullptr;
    if (oL1 != Py_None) {
        const at::Tensor *L1 = plain_tensor(oL1), *L2 = plain_tensor(oL2);
        if (!L1 || !L2 || L1->dim() != 2 || L2->dim() != 2 || L1->size(1) < 1 || L1->size(1) > INT_MAX) Py_RETURN_NONE;
        if (L1->scalar_type() != at::kBFloat16 || L2->scalar_type() != at::kBFloat16 || !L1->is_contiguous() || !L2->is_contiguous()) Py_RETURN_NONE;
        r = static_cast<int>(L1->size(1));
        if (L1->size(0) != N || L2->size(0) != r || L2->size(1) != K) Py_RETURN_NONE;
        L1p = L1->data_ptr(); L2p = L2->data_ptr();
    } else if (oL2 != Py_None) {
        Py_RETURN_NONE;
    }
    const int64_t M = A->size(0);
    at::Tensor fresh;
    void* out;
    if (oout == Py_None) {
        fresh = at::empty({M, backward ? K : N}, A->options());
        if (!plain(fresh)) Py_RETURN_NONE;
        out = fresh.data_ptr();
    } else {
        const at::Tensor* given = plain_tensor(oout);
        if (!given) Py_RETURN_NONE;
        out = given->data_ptr();
    }
    const void* a = A->data_ptr();
    void* w = ws->data_ptr();
    const size_t w_bytes = static_cast<size_t>(ws->numel());
    void* stream = c10::cuda::getCurrentCUDAStream().stream();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = g_linear[backward ? 1 : 0](&m, L1p, L2p, r, a, M, out, w, w_bytes, stream);
    Py_END_ALLOW_THREADS
    if (rc != LQLORA_OK) return PyLong_FromLong(rc);
    if (oout != Py_None) { Py_INCREF(oout); return oout; }
    return THPVariable_Wrap(std::move(fresh));
    END_HANDLE_TH_ERRORS
}

// encode(W, cfg, workspace) -> (codes, scale codes, second-level scales), status number of a call that failed, or None.
PyObject* encode(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 3 || !g_qmatrix || modes()) Py_RETURN_NONE;
    if (reinterpret_cast<PyObject*>(Py_TYPE(args[0])) != THPVariableClass) Py_RETURN_NONE;
    const at::Tensor* W = plain_tensor(args[0]);
    if (!W || W->scalar_type() != at::kFloat || W->dim() != 2 || !W->is_contiguous()) Py_RETURN_NONE;
    lqlora_qmatrix m{};
    if (!config_of(args[1], &m.cfg) || m.cfg.b1 != 8 || m.cfg.b2 != 32) Py_RETURN_NONE;
    m.N = W->size(0); m.K = W->size(1);
    size_t code_bytes, scale_bytes, scale2_bytes, ws_bytes;
    if (g_sizes(m.N, m.K, &m.cfg, &code_bytes, &scale_bytes, &scale2_bytes, &ws_bytes) != LQLORA_OK) Py_RETURN_NONE;
    at::Tensor scratch;
    const at::Tensor* ws = &scratch;
    const auto bytes = W->options().dtype(at::kByte);
    if (args[2] != Py_None) {
        ws = plain_tensor(args[2]);
        if (!ws) Py_RETURN_NONE;
    } else {
        scratch = at::empty({static_cast<int64_t>(ws_bytes < 16 ? 16 : ws_bytes)}, bytes);
    }
    at::Tensor codes = at::empty({static_cast<int64_t>(code_bytes)}, bytes), sc = at::empty({static_cast<int64_t>(scale_bytes)}, bytes),
               s2 = at::empty({static_cast<int64_t>(scale2_bytes / 4)}, W->options());
    if (!plain(*ws) || !plain(codes) || !plain(sc) || !plain(s2)) Py_RETURN_NONE;
    m.codes = codes.data_ptr(); m.scale_codes = static_cast<uint8_t*>(sc.data_ptr()); m.scale2 = static_cast<float*>(s2.data_ptr());
    const float* src = static_cast<const float*>(W->data_ptr());
    void* w = ws->data_ptr();
    const size_t w_bytes = static_cast<size_t>(ws->numel());
    void* stream = c10::cuda::getCurrentCUDAStream().stream();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = g_encode(src, &m, w, w_bytes, stream);
    Py_END_ALLOW_THREADS
    if (rc != LQLORA_OK) return PyLong_FromLong(rc);
    PyObject* parts[3] = {THPVariable_Wrap(std::move(codes)), THPVariable_Wrap(std::move(sc)), THPVariable_Wrap(std::move(s2))};
    PyObject* out = parts[0] && parts[1] && parts[2] ? PyTuple_Pack(3, parts[0], parts[1], parts[2]) : nullptr;
    for (PyObject* p : parts) Py_XDECREF(p);
    return out;
    END_HANDLE_TH_ERRORS
}

// setup(addresses of lqlora_linear_fwd, lqlora_linear_bwd_input, lqlora_packed_sizes, lqlora_encode; torch.nn.Parameter, QMatrix)
PyObject* setup(PyObject*, PyObject* args) {
    unsigned long long f, b, s, e;
    PyObject *parameter, *qmatrix;
    if (!PyArg_ParseTuple(args, "KKKKOO", &f, &b, &s, &e, &parameter, &qmatrix)) return nullptr;
    g_linear[0] = reinterpret_cast<LinearFn>(f);
    g_linear[1] = reinterpret_cast<LinearFn>(b);
    g_sizes = reinterpret_cast<SizesFn>(s);
    g_encode = reinterpret_cast<EncodeFn>(e);
    Py_INCREF(parameter); Py_INCREF(qmatrix);
    Py_XSETREF(g_parameter, parameter);
    Py_XSETREF(g_qmatrix, qmatrix);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"linear", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(linear)), METH_FASTCALL, nullptr},
    {"encode", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(encode)), METH_FASTCALL, nullptr},
    {"setup", setup, METH_VARARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fast", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fast(void) {
    s_codes = PyUnicode_InternFromString("codes"); s_scale_codes = PyUnicode_InternFromString("scale_codes"); s_scale2 = PyUnicode_InternFromString("scale2");
    s_N = PyUnicode_InternFromString("N"); s_K = PyUnicode_InternFromString("K"); s_cfg = PyUnicode_InternFromString("cfg");
    s_b0 = PyUnicode_InternFromString("b0"); s_B0 = PyUnicode_InternFromString("B0"); s_b1 = PyUnicode_InternFromString("b1");
    s_B1 = PyUnicode_InternFromString("B1"); s_b2 = PyUnicode_InternFromString("b2");
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", LQLORA_BUILT_FOR) != 0) { Py_DECREF(m); return nullptr; }
    return m;
}
