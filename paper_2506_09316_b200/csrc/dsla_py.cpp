// Argument marshalling of the per-token and per-prompt entry points for Python, as a CPython extension (module _native).
// A decode step of a few rows takes the GPU about as long as filling a ctypes structure takes the interpreter: reading
// data pointers, shapes and the current stream through the C++ side of torch costs well under a microsecond per call
// (a decode step of one row, back to back: 10.7 us through ctypes).
// Nothing is computed here; every function fills the argument structure of include/dsla.h, calls the C
// entry point of the same name and returns its status.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>

#include "dsla.h"

namespace {

// The tensor behind a Python argument: nullptr for None (and with an exception set for anything else).
struct Arg {
    const at::Tensor* t = nullptr;
    void* ptr = nullptr;
};
bool read_tensor(PyObject* o, Arg* out) {
    if (o == Py_None) return true;
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "expected a torch tensor or None, got %s", Py_TYPE(o)->tp_name);
        return false;
    }
    out->t = &THPVariable_Unpack(o);
    out->ptr = out->t->data_ptr();
    return true;
}
bool read_tensors(PyObject* const* args, int n, Arg* out) {
    for (int i = 0; i < n; ++i)
        if (!read_tensor(args[i], &out[i])) return false;
    return true;
}
bool has_dims(const Arg& a, int dims, const char* name) {
    if (a.t && a.t->dim() == dims) return true;
    PyErr_Format(PyExc_ValueError, "%s must be a tensor of %d dimensions", name, dims);
    return false;
}
bool has_dims_from(const Arg& a, int dims, const char* name) {      // further dimensions are the caller's business: only size(dims - 1) is read
    if (a.t && a.t->dim() >= dims) return true;
    PyErr_Format(PyExc_ValueError, "%s must be a tensor of at least %d dimensions", name, dims);
    return false;
}
bool read_dtype(const at::Tensor& t, dsla_dtype* out) {
    if (t.scalar_type() == at::kBFloat16) { *out = DSLA_BF16; return true; }
    if (t.scalar_type() == at::kFloat) { *out = DSLA_F32; return true; }
    PyErr_SetString(PyExc_KeyError, "the element type must be torch.float32 or torch.bfloat16");
    return false;
}
dsla_gate_layout layout_of(const Arg& gates, int scalar_dims) {
    return gates.t && gates.t->dim() == scalar_dims + 1 ? DSLA_GATE_PER_KEY_CHANNEL : DSLA_GATE_SCALAR;
}
bool read_int(PyObject* o, int* out) {
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) return false;
    if (v != (int)v) { PyErr_SetString(PyExc_OverflowError, "value does not fit a C int"); return false; }
    *out = (int)v;
    return true;
}
bool read_float(PyObject* o, float* out) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) return false;
    *out = (float)v;
    return true;
}
bool read_handle(PyObject* o, dsla_state** out) {
    *out = o == Py_None ? nullptr : static_cast<dsla_state*>(PyLong_AsVoidPtr(o));
    return !PyErr_Occurred();
}
bool read_stream(PyObject* o, void** out) {
    if (o == Py_None) *out = c10::cuda::getCurrentCUDAStream().stream();
    else *out = PyLong_AsVoidPtr(o);
    return !PyErr_Occurred();
}
bool count_is(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return false;
}
size_t nbytes_of(const Arg& a) { return a.t ? (size_t)a.t->numel() * (size_t)a.t->element_size() : 0; }

// Runs a C entry point without the interpreter lock (a launch can wait for room in the stream's queue).
template <typename F> PyObject* status_of(F call) {
    dsla_status rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

#define GUARD_BEGIN try {
#define GUARD_END                                      \
    } catch (const std::exception& e) {                \
        PyErr_SetString(PyExc_RuntimeError, e.what()); \
        return nullptr;                                \
    }

// decode_step(q, k, v, o, g_hist, g_rec, gamma, slots, row_mask, handle, scale, stream) -> status
PyObject* py_decode_step(PyObject*, PyObject* const* args, Py_ssize_t n) {
    GUARD_BEGIN
    Arg t[9];
    dsla_state* st;
    void* stream;
    dsla_decode_args a;
    std::memset(&a, 0, sizeof(a));
    if (!count_is(n, 12) || !read_tensors(args, 9, t) || !has_dims(t[0], 3, "q") || !has_dims_from(t[2], 3, "v") ||
        !read_dtype(*t[0].t, &a.dtype) || !read_handle(args[9], &st) || !read_float(args[10], &a.scale) || !read_stream(args[11], &stream))
        return nullptr;
    a.q = t[0].ptr; a.k = t[1].ptr; a.v = t[2].ptr; a.o = t[3].ptr;
    a.g_hist = static_cast<float*>(t[4].ptr); a.g_rec = static_cast<float*>(t[5].ptr); a.gamma = static_cast<float*>(t[6].ptr);
    a.slots = static_cast<int32_t*>(t[7].ptr); a.row_mask = static_cast<uint8_t*>(t[8].ptr);
    a.B = (int)t[0].t->size(0); a.H = (int)t[0].t->size(1); a.d_k = (int)t[0].t->size(2); a.d_v = (int)t[2].t->size(2);
    a.gate_layout = layout_of(t[4], 2);
    return status_of([&] { return dsla_decode_step(&a, st, stream); });
    GUARD_END
}

// nstate_decode_step(q, k, v, o, gates, weights, slots, row_mask, handle, scale, stream) -> status
PyObject* py_nstate_decode_step(PyObject*, PyObject* const* args, Py_ssize_t n) {
    GUARD_BEGIN
    Arg t[8];
    dsla_state* st;
    void* stream;
    dsla_nstate_decode_args a;
    std::memset(&a, 0, sizeof(a));
    if (!count_is(n, 11) || !read_tensors(args, 8, t) || !has_dims(t[0], 3, "q") || !has_dims_from(t[2], 3, "v") || !read_dtype(*t[0].t, &a.dtype) ||
        !read_handle(args[8], &st) || !read_float(args[9], &a.scale) || !read_stream(args[10], &stream))
        return nullptr;
    if (!t[4].t || t[4].t->dim() < 1) { PyErr_SetString(PyExc_ValueError, "gates must be a tensor"); return nullptr; }
    a.q = t[0].ptr; a.k = t[1].ptr; a.v = t[2].ptr; a.o = t[3].ptr;
    a.gates = static_cast<float*>(t[4].ptr); a.weights = static_cast<float*>(t[5].ptr);
    a.slots = static_cast<int32_t*>(t[6].ptr); a.row_mask = static_cast<uint8_t*>(t[7].ptr);
    a.B = (int)t[0].t->size(0); a.H = (int)t[0].t->size(1); a.d_k = (int)t[0].t->size(2); a.d_v = (int)t[2].t->size(2);
    a.n_states = (int)t[4].t->size(0);
    a.gate_layout = layout_of(t[4], 3);
    return status_of([&] { return dsla_nstate_decode_step(&a, st, stream); });
    GUARD_END
}

// prefill(q, k, v, o, g_hist, g_rec, gamma, cu_seqlens, slots, workspace, handle, N, T, max_seqlen, chunk, scale,
//         use_initial_state, impl, stream) -> status
PyObject* py_prefill(PyObject*, PyObject* const* args, Py_ssize_t n) {
    GUARD_BEGIN
    Arg t[10];
    dsla_state* st;
    void* stream;
    int impl;
    dsla_prefill_args a;
    std::memset(&a, 0, sizeof(a));
    if (!count_is(n, 19) || !read_tensors(args, 10, t) || !has_dims(t[0], 3, "q") || !has_dims_from(t[2], 3, "v") || !read_dtype(*t[0].t, &a.dtype) ||
        !read_handle(args[10], &st) || !read_int(args[11], &a.N) || !read_int(args[12], &a.T) || !read_int(args[13], &a.max_seqlen) ||
        !read_int(args[14], &a.chunk) || !read_float(args[15], &a.scale) || !read_int(args[16], &a.use_initial_state) ||
        !read_int(args[17], &impl) || !read_stream(args[18], &stream))
        return nullptr;
    a.q = t[0].ptr; a.k = t[1].ptr; a.v = t[2].ptr; a.o = t[3].ptr;
    a.g_hist = static_cast<float*>(t[4].ptr); a.g_rec = static_cast<float*>(t[5].ptr); a.gamma = static_cast<float*>(t[6].ptr);
    a.cu_seqlens = static_cast<int32_t*>(t[7].ptr); a.slots = static_cast<int32_t*>(t[8].ptr);
    a.workspace = t[9].ptr; a.workspace_bytes = nbytes_of(t[9]);
    a.T_total = (int)t[0].t->size(0); a.H = (int)t[0].t->size(1); a.d_k = (int)t[0].t->size(2); a.d_v = (int)t[2].t->size(2);
    a.impl = static_cast<dsla_impl>(impl);
    a.gate_layout = layout_of(t[4], 2);
    return status_of([&] { return dsla_prefill(&a, st, stream); });
    GUARD_END
}

// Sizes, types and layouts of a prefill call, which is all that its workspace depends on.
bool read_sizes(PyObject* const* args, const Arg& q, const Arg& v, const Arg& cu, dsla_prefill_args* a) {
    if (!has_dims(q, 3, "q") || !has_dims_from(v, 3, "v") || !read_dtype(*q.t, &a->dtype) || !read_int(args[0], &a->N) || !read_int(args[1], &a->T) ||
        !read_int(args[2], &a->max_seqlen))
        return false;
    a->cu_seqlens = static_cast<int32_t*>(cu.ptr);
    a->T_total = (int)q.t->size(0); a->H = (int)q.t->size(1); a->d_k = (int)q.t->size(2); a->d_v = (int)v.t->size(2);
    a->scale = 1.f;
    return true;
}

// prefill_workspace(q, v, g_hist, cu_seqlens, N, T, max_seqlen, chunk, impl) -> bytes
PyObject* py_prefill_workspace(PyObject*, PyObject* const* args, Py_ssize_t n) {
    GUARD_BEGIN
    Arg t[4];
    int impl;
    dsla_prefill_args a;
    std::memset(&a, 0, sizeof(a));
    if (!count_is(n, 9) || !read_tensors(args, 4, t) || !read_sizes(args + 4, t[0], t[1], t[3], &a) || !read_int(args[7], &a.chunk) || !read_int(args[8], &impl))
        return nullptr;
    a.impl = static_cast<dsla_impl>(impl);
    a.gate_layout = layout_of(t[2], 2);
    return PyLong_FromSize_t(dsla_prefill_workspace_bytes(&a));
    GUARD_END
}

// nstate_prefill_workspace(q, v, gates, cu_seqlens, N, T, max_seqlen, impl) -> bytes
PyObject* py_nstate_prefill_workspace(PyObject*, PyObject* const* args, Py_ssize_t n) {
    GUARD_BEGIN
    Arg t[4];
    int impl;
    dsla_prefill_args s;
    std::memset(&s, 0, sizeof(s));
    if (!count_is(n, 8) || !read_tensors(args, 4, t) || !read_sizes(args + 4, t[0], t[1], t[3], &s) || !read_int(args[7], &impl)) return nullptr;
    if (!t[2].t || t[2].t->dim() < 1) { PyErr_SetString(PyExc_ValueError, "gates must be a tensor"); return nullptr; }
    dsla_nstate_prefill_args a;
    std::memset(&a, 0, sizeof(a));
    a.cu_seqlens = s.cu_seqlens; a.N = s.N; a.T = s.T; a.T_total = s.T_total; a.max_seqlen = s.max_seqlen;
    a.H = s.H; a.d_k = s.d_k; a.d_v = s.d_v; a.dtype = s.dtype; a.scale = 1.f;
    a.n_states = (int)t[2].t->size(0);
    a.impl = static_cast<dsla_impl>(impl);
    a.gate_layout = layout_of(t[2], 3);
    return PyLong_FromSize_t(dsla_nstate_prefill_workspace_bytes(&a));
    GUARD_END
}

// nstate_prefill(q, k, v, o, gates, weights, cu_seqlens, slots, workspace, handle, N, T, max_seqlen, scale,
//                use_initial_state, impl, stream) -> status
PyObject* py_nstate_prefill(PyObject*, PyObject* const* args, Py_ssize_t n) {
    GUARD_BEGIN
    Arg t[9];
    dsla_state* st;
    void* stream;
    int impl;
    dsla_nstate_prefill_args a;
    std::memset(&a, 0, sizeof(a));
    if (!count_is(n, 17) || !read_tensors(args, 9, t) || !has_dims(t[0], 3, "q") || !has_dims_from(t[2], 3, "v") || !read_dtype(*t[0].t, &a.dtype) ||
        !read_handle(args[9], &st) || !read_int(args[10], &a.N) || !read_int(args[11], &a.T) || !read_int(args[12], &a.max_seqlen) ||
        !read_float(args[13], &a.scale) || !read_int(args[14], &a.use_initial_state) || !read_int(args[15], &impl) ||
        !read_stream(args[16], &stream))
        return nullptr;
    if (!t[4].t || t[4].t->dim() < 1) { PyErr_SetString(PyExc_ValueError, "gates must be a tensor"); return nullptr; }
    a.q = t[0].ptr; a.k = t[1].ptr; a.v = t[2].ptr; a.o = t[3].ptr;
    a.gates = static_cast<float*>(t[4].ptr); a.weights = static_cast<float*>(t[5].ptr);
    a.cu_seqlens = static_cast<int32_t*>(t[6].ptr); a.slots = static_cast<int32_t*>(t[7].ptr);
    a.workspace = t[8].ptr; a.workspace_bytes = nbytes_of(t[8]);
    a.T_total = (int)t[0].t->size(0); a.H = (int)t[0].t->size(1); a.d_k = (int)t[0].t->size(2); a.d_v = (int)t[2].t->size(2);
    a.n_states = (int)t[4].t->size(0);
    a.impl = static_cast<dsla_impl>(impl);
    a.gate_layout = layout_of(t[4], 3);
    return status_of([&] { return dsla_nstate_prefill(&a, st, stream); });
    GUARD_END
}

// gate_project(x, w, bias, g_hist, g_rec, stream) -> status
PyObject* py_gate_project(PyObject*, PyObject* const* args, Py_ssize_t n) {
    GUARD_BEGIN
    Arg t[5];
    void* stream;
    dsla_gate_project_args a;
    std::memset(&a, 0, sizeof(a));
    if (!count_is(n, 6) || !read_tensors(args, 5, t) || !has_dims(t[0], 2, "x") || !has_dims_from(t[1], 1, "w") || !read_stream(args[5], &stream)) return nullptr;
    a.x = t[0].ptr; a.w = t[1].ptr; a.bias = static_cast<float*>(t[2].ptr);
    a.g_hist = static_cast<float*>(t[3].ptr); a.g_rec = static_cast<float*>(t[4].ptr);
    a.T = (int)t[0].t->size(0); a.D_model = (int)t[0].t->size(1); a.H = (int)(t[1].t->size(0) / 2);
    return status_of([&] { return dsla_gate_project(&a, stream); });
    GUARD_END
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f))
PyMethodDef kMethods[] = {{"decode_step", FAST(py_decode_step), METH_FASTCALL, nullptr},
                          {"nstate_decode_step", FAST(py_nstate_decode_step), METH_FASTCALL, nullptr},
                          {"prefill", FAST(py_prefill), METH_FASTCALL, nullptr},
                          {"prefill_workspace", FAST(py_prefill_workspace), METH_FASTCALL, nullptr},
                          {"nstate_prefill_workspace", FAST(py_nstate_prefill_workspace), METH_FASTCALL, nullptr},
                          {"nstate_prefill", FAST(py_nstate_prefill), METH_FASTCALL, nullptr},
                          {"gate_project", FAST(py_gate_project), METH_FASTCALL, nullptr},
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", "Argument marshalling of libdsla for torch tensors.", -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&kModule); }
