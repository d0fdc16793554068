// Argument marshalling of the calls a control loop makes many times per tick, for binding.py: tensors and scalars in, the status code of
// the C ABI out (include/reflex.h). What bounds a small direct call is the host: the launch itself is some 3.3 us, and pulling
// pointers, sizes and the stream out of the tensors in Python and through ctypes took another 2 to 3. No arithmetic, no state.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <vector>

#include "reflex.h"

namespace {

struct Bad {};      // a Python exception is set

const at::Tensor &tensor(PyObject *o)
{
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a torch tensor");
        throw Bad();
    }
    return THPVariable_Unpack(o);
}

void *ptr(PyObject *o)
{
    if (o == Py_None) return nullptr;
    const at::Tensor &t = tensor(o);
    if (!t.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "tensor must be contiguous");
        throw Bad();
    }
    return t.data_ptr();
}

int dtype(PyObject *o)
{
    const at::Tensor &t = tensor(o);
    if (t.scalar_type() == at::kBFloat16) return REFLEX_DTYPE_BF16;
    if (t.scalar_type() == at::kFloat) return REFLEX_DTYPE_F32;
    PyErr_SetString(PyExc_ValueError, "unsupported storage dtype");
    throw Bad();
}

int dim(PyObject *o, int i)
{
    const at::Tensor &t = tensor(o);
    if (i < 0) i += (int)t.dim();
    if (i < 0 || i >= t.dim()) {
        PyErr_SetString(PyExc_ValueError, "tensor has too few dimensions");
        throw Bad();
    }
    return (int)t.size(i);
}

void want_dims(PyObject *o, int n)
{
    if (tensor(o).dim() != n) {
        PyErr_Format(PyExc_ValueError, "expected a tensor of %d dimensions, got %d", n, (int)tensor(o).dim());
        throw Bad();
    }
}

int integer(PyObject *o)
{
    // (anything int() takes, as the Python binding did)
    PyObject *n = PyLong_Check(o) ? (Py_INCREF(o), o) : PyNumber_Long(o);
    if (!n) throw Bad();
    const long v = PyLong_AsLong(n);
    Py_DECREF(n);
    if (v == -1 && PyErr_Occurred()) throw Bad();
    return (int)v;
}

float real(PyObject *o)
{
    // (anything float() takes)
    PyObject *n = PyFloat_Check(o) ? (Py_INCREF(o), o) : PyNumber_Float(o);
    if (!n) throw Bad();
    const double v = PyFloat_AS_DOUBLE(n);
    Py_DECREF(n);
    return (float)v;
}

reflex_cache_t *handle(PyObject *o)      // the handle as an integer, 0 or None = NULL
{
    if (o == Py_None) return nullptr;
    void *p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) throw Bad();
    return (reflex_cache_t *)p;
}

void *stream(PyObject *o)                // None: torch's current stream; else a torch stream or a stream handle
{
    if (o == Py_None) return (void *)c10::cuda::getCurrentCUDAStream().stream();
    PyObject *v = PyLong_Check(o) ? (Py_INCREF(o), o) : PyObject_GetAttrString(o, "cuda_stream");
    if (!v) { PyErr_Clear(); v = PyNumber_Long(o); }
    if (!v) throw Bad();
    void *p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (!p && PyErr_Occurred()) throw Bad();
    return p;
}

std::vector<int32_t> ints(PyObject *o)
{
    std::vector<int32_t> v;
    if (o == Py_None) return v;
    PyObject *seq = PySequence_Fast(o, "expected a sequence of integers");
    if (!seq) throw Bad();
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    v.reserve((size_t)(n > 0 ? n : 1));      // (no elements is not the same as no list: data() is not NULL)
    try {
        for (Py_ssize_t i = 0; i < n; ++i) v.push_back(integer(PySequence_Fast_GET_ITEM(seq, i)));
    } catch (...) { Py_DECREF(seq); throw; }
    Py_DECREF(seq);
    return v;
}

// The call runs without the interpreter lock (a launch may block when the device's queue is full), which is taken again whatever way
// the call ends.
template <typename F>
int unlocked(F &&f)
{
    struct Unlocked {
        PyThreadState *state = PyEval_SaveThread();
        ~Unlocked() { PyEval_RestoreThread(state); }
    } guard;
    return f();
}

template <typename F>
PyObject *entry(Py_ssize_t got, Py_ssize_t want, F &&f)
{
    if (got != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
        return nullptr;
    }
    try {
        return f();
    } catch (const Bad &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// x, y, cond, W1, b1, W2, b2, gate_buf, eps, stream
PyObject *adarmsnorm(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return entry(n, 10, [&]() -> PyObject * {
        want_dims(a[0], 3);
        if (a[3] != Py_None) want_dims(a[3], 2);
        const int B = dim(a[0], 0), R = dim(a[0], 1), D = dim(a[0], 2), Hd = a[3] == Py_None ? 0 : dim(a[3], 0), Cd = a[3] == Py_None ? 0 : dim(a[3], 1);
        const int dt = dtype(a[0]);
        const float eps = real(a[8]);
        void *p[8];
        for (int i = 0; i < 8; ++i) p[i] = ptr(a[i]);
        void *st = stream(a[9]);
        return PyLong_FromLong(unlocked([&] { return reflex_adarmsnorm(p[0], p[1], p[2], p[3], p[4], p[5], p[6], (float *)p[7], B, R, D, Cd, Hd, eps, dt, st); }));
    });
}

// cond, W1, b1, W2, b2, gate_buf, stream
PyObject *adarmsnorm_gate(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return entry(n, 7, [&]() -> PyObject * {
        want_dims(a[0], 2);
        const int B = dim(a[0], 0), Cd = dim(a[0], 1), L = tensor(a[1]).dim() == 3 ? dim(a[1], 0) : 1, D = dim(a[3], -2), Hd = dim(a[1], -2), dt = dtype(a[0]);
        void *p[6];
        for (int i = 0; i < 6; ++i) p[i] = ptr(a[i]);
        void *st = stream(a[6]);
        return PyLong_FromLong(unlocked([&] { return reflex_adarmsnorm_gate(p[0], p[1], p[2], p[3], p[4], (float *)p[5], L, B, D, Cd, Hd, dt, st); }));
    });
}

// handle, x, gate, Wqkv, q, k_dyn, v_dyn, eps, impl, stream
PyObject *adarmsnorm_qkv(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return entry(n, 10, [&]() -> PyObject * {
        want_dims(a[1], 3);
        const int B = dim(a[1], 0), R = dim(a[1], 1), D = dim(a[1], 2), Hq = dim(a[4], 2), d = dim(a[4], 3), Hkv = dim(a[5], 2), dt = dtype(a[1]), impl = integer(a[8]);
        const float eps = real(a[7]);
        reflex_cache_t *c = handle(a[0]);
        void *p[7];
        for (int i = 1; i < 7; ++i) p[i] = ptr(a[i]);
        void *st = stream(a[9]);
        return PyLong_FromLong(unlocked([&] { return reflex_adarmsnorm_qkv(c, p[1], (const float *)p[2], p[3], p[4], p[5], p[6], B, R, D, Hq, Hkv, d, eps, dt, impl, st); }));
    });
}

// handle, x, gate, Wgu, h, eps, impl, stream
PyObject *adarmsnorm_swiglu(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return entry(n, 8, [&]() -> PyObject * {
        want_dims(a[1], 3);
        const int B = dim(a[1], 0), R = dim(a[1], 1), D = dim(a[1], 2), F = dim(a[4], 2), dt = dtype(a[1]), impl = integer(a[6]);
        const float eps = real(a[5]);
        reflex_cache_t *c = handle(a[0]);
        void *p[5];
        for (int i = 1; i < 5; ++i) p[i] = ptr(a[i]);
        void *st = stream(a[7]);
        return PyLong_FromLong(unlocked([&] { return reflex_adarmsnorm_swiglu(c, p[1], (const float *)p[2], p[3], p[4], B, R, D, F, eps, dt, impl, st); }));
    });
}

// handle, a, W, res, out, impl, stream
PyObject *linear_residual(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return entry(n, 7, [&]() -> PyObject * {
        const int K = dim(a[1], -1), N = dim(a[2], 0), M = K > 0 ? (int)(tensor(a[1]).numel() / K) : 0, dt = dtype(a[1]), impl = integer(a[5]);
        reflex_cache_t *c = handle(a[0]);
        void *p[5];
        for (int i = 1; i < 5; ++i) p[i] = ptr(a[i]);
        void *st = stream(a[6]);
        return PyLong_FromLong(unlocked([&] { return reflex_linear_residual(c, p[1], p[2], p[3], p[4], M, K, N, dt, impl, st); }));
    });
}

// handle, layer, q, k_dyn, v_dyn, out, scale, dyn_mask, stream
PyObject *partitioned_attention(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return entry(n, 9, [&]() -> PyObject * {
        reflex_cache_t *c = handle(a[0]);
        const int layer = integer(a[1]), T = dim(a[2], 1), mask = integer(a[7]);
        const float scale = real(a[6]);
        void *p[6];
        for (int i = 2; i < 6; ++i) p[i] = ptr(a[i]);
        void *st = stream(a[8]);
        return PyLong_FromLong(unlocked([&] { return reflex_partitioned_attention(c, layer, p[2], p[3], p[4], p[5], T, scale, mask, st); }));
    });
}

// x, v, x_lowp, k, K, stream
PyObject *flow_step(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return entry(n, 6, [&]() -> PyObject * {
        want_dims(a[0], 3);
        const int B = dim(a[0], 0), T = dim(a[0], 1), A = dim(a[0], 2), k = integer(a[3]), K = integer(a[4]), dt = dtype(a[1]);
        void *x = ptr(a[0]), *v = ptr(a[1]), *lowp = ptr(a[2]), *st = stream(a[5]);
        return PyLong_FromLong(unlocked([&] { return reflex_flow_step(x, v, lowp, B, T, A, k, K, dt, st); }));
    });
}

// which (0 init, 1 stage), handle, stream_ids, k_static, v_static, S or None, stream
PyObject *write_static(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return entry(n, 7, [&]() -> PyObject * {
        const int which = integer(a[0]), S_src = a[3] == Py_None ? 0 : dim(a[3], 2);
        reflex_cache_t *c = handle(a[1]);
        const std::vector<int32_t> ids = ints(a[2]), S = ints(a[5]);
        if (a[5] != Py_None && S.size() < ids.size()) {
            PyErr_SetString(PyExc_ValueError, "a prefix length for every stream");
            throw Bad();
        }
        void *k = ptr(a[3]), *v = ptr(a[4]), *st = stream(a[6]);
        const int32_t *Sp = a[5] == Py_None ? nullptr : S.data();
        return PyLong_FromLong(unlocked([&] {
            return which ? reflex_cache_stage_static(c, ids.data(), (int)ids.size(), k, v, S_src, Sp, st) : reflex_cache_init_static(c, ids.data(), (int)ids.size(), k, v, S_src, Sp, st);
        }));
    });
}

// handle, stream_ids, stream
PyObject *commit_static(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return entry(n, 3, [&]() -> PyObject * {
        reflex_cache_t *c = handle(a[0]);
        const std::vector<int32_t> ids = ints(a[1]);
        void *st = stream(a[2]);
        return PyLong_FromLong(unlocked([&] { return reflex_cache_commit_static(c, ids.data(), (int)ids.size(), st); }));
    });
}

// handle, stream_ids, k_new, v_new, stream -> status code, or the list of eviction counts
PyObject *append_sliding(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return entry(n, 5, [&]() -> PyObject * {
        reflex_cache_t *c = handle(a[0]);
        const std::vector<int32_t> ids = ints(a[1]);
        const int m = dim(a[2], 2);
        void *k = ptr(a[2]), *v = ptr(a[3]), *st = stream(a[4]);
        std::vector<int32_t> ev(ids.size());
        const int rc = unlocked([&] { return reflex_cache_append_sliding(c, ids.data(), (int)ids.size(), k, v, m, ev.data(), st); });
        if (rc != REFLEX_OK) return PyLong_FromLong(rc);
        PyObject *out = PyList_New((Py_ssize_t)ev.size());
        if (!out) throw Bad();
        for (size_t i = 0; i < ev.size(); ++i) PyList_SET_ITEM(out, (Py_ssize_t)i, PyLong_FromLong(ev[i]));
        return out;
    });
}

#define M(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {M(adarmsnorm), M(adarmsnorm_gate), M(adarmsnorm_qkv), M(adarmsnorm_swiglu), M(linear_residual), M(partitioned_attention), M(flow_step),
                         M(write_static), M(commit_static), M(append_sliding), {nullptr, nullptr, 0, nullptr}};
#undef M
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void) { return PyModule_Create(&module); }
