// Python entry points of the calls a program makes per token, layer or step: the same names and argument
// order as binding.py's, marshalled natively.  A generation step is a 7-12 us kernel; marshalling its
// twelve tensors through ctypes and asking torch for the current stream in Python took 13-16 us per call and
// set the pace of small batches.  Here a tensor argument is checked (device-resident, contiguous),
// unwrapped and passed on without an intermediate Python object.
#include <Python.h>
#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>

#include "../../include/natsl.h"

namespace {

// Arguments of one call, in order; `ok` goes false with a Python error set.
struct Args {
    PyObject *const *v;
    bool ok = true;

    const at::Tensor *tensor(int i) {
        if (!ok) return nullptr;
        if (v[i] == Py_None) return nullptr;
        if (!THPVariable_Check(v[i])) {
            PyErr_Format(PyExc_TypeError, "argument %d: a tensor or None is expected", i);
            ok = false;
            return nullptr;
        }
        const at::Tensor &t = THPVariable_Unpack(v[i]);
        if (!t.is_cuda() || !t.is_contiguous()) {
            PyErr_SetString(PyExc_AssertionError, "device-resident contiguous tensors only");
            ok = false;
            return nullptr;
        }
        return &t;
    }
    template <typename T> T *ptr(int i) {
        const at::Tensor *t = tensor(i);
        return t ? static_cast<T *>(t->data_ptr()) : nullptr;
    }
    size_t numel(int i) {
        const at::Tensor *t = tensor(i);
        return t ? static_cast<size_t>(t->numel()) : 0;
    }
    int64_t size(int i, int dim) {
        const at::Tensor *t = tensor(i);
        if (t && (dim < 0 ? t->dim() < -dim : t->dim() <= dim)) {
            PyErr_Format(PyExc_IndexError, "argument %d: too few dimensions", i);
            ok = false;
        }
        return t && ok ? t->size(dim) : 0;
    }
    long integer(int i) {
        if (!ok) return 0;
        const long x = PyLong_AsLong(v[i]);
        if (x == -1 && PyErr_Occurred()) ok = false;
        return x;
    }
    const natsl_params *params(int i) {      // a ctypes natsl_params, through the buffer protocol
        if (!ok) return nullptr;
        Py_buffer b;
        if (PyObject_GetBuffer(v[i], &b, PyBUF_SIMPLE) != 0) { ok = false; return nullptr; }
        const void *p = b.buf;
        if (b.len != (Py_ssize_t)sizeof(natsl_params)) {
            PyErr_SetString(PyExc_TypeError, "natsl_params expected");
            ok = false;
        }
        PyBuffer_Release(&b);                // (the caller's argument keeps the structure alive)
        return ok ? static_cast<const natsl_params *>(p) : nullptr;
    }
};

bool current_stream(void **st) {
    try {
        *st = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return false;
    }
}

bool count_is(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, n);
    return false;
}

// (the call itself only enqueues work, but may wait for the library's enqueue mutex: without the GIL)
#define NATSL_CALL(expr)                          \
    void *st;                                     \
    if (!a.ok || !current_stream(&st)) return nullptr; \
    int rc;                                       \
    Py_BEGIN_ALLOW_THREADS rc = (expr);           \
    Py_END_ALLOW_THREADS                          \
    return PyLong_FromLong(rc)

PyObject *hybrid_fwd(PyObject *, PyObject *const *v, Py_ssize_t n) {
    if (!count_is(n, 9)) return nullptr;
    Args a{v};
    const void *q = a.ptr<void>(0), *k = a.ptr<void>(1), *vv = a.ptr<void>(2);
    const float *g = a.ptr<float>(3), *beta = a.ptr<float>(4);
    const uint8_t *route = a.ptr<uint8_t>(5);
    void *out = a.ptr<void>(6), *ws = a.ptr<void>(8);
    const natsl_params *p = a.params(7);
    const size_t wb = a.numel(8);
    NATSL_CALL(natsl_hybrid_fwd(q, k, vv, g, beta, route, out, p, ws, wb, st));
}

PyObject *hybrid_fwd_static(PyObject *, PyObject *const *v, Py_ssize_t n) {
    if (!count_is(n, 8)) return nullptr;
    Args a{v};
    const void *q = a.ptr<void>(0), *k = a.ptr<void>(1), *vv = a.ptr<void>(2);
    const float *g = a.ptr<float>(3), *beta = a.ptr<float>(4);
    const uint8_t *route = a.ptr<uint8_t>(5);
    void *out = a.ptr<void>(6);
    const natsl_params *p = a.params(7);
    NATSL_CALL(natsl_hybrid_fwd_static(q, k, vv, g, beta, route, out, p, st));
}

PyObject *hybrid_bwd(PyObject *, PyObject *const *v, Py_ssize_t n) {
    if (!count_is(n, 15)) return nullptr;
    Args a{v};
    const void *q = a.ptr<void>(0), *k = a.ptr<void>(1), *vv = a.ptr<void>(2);
    const float *g = a.ptr<float>(3), *beta = a.ptr<float>(4);
    const uint8_t *route = a.ptr<uint8_t>(5);
    const void *dout = a.ptr<void>(6);
    void *dq = a.ptr<void>(7), *dk = a.ptr<void>(8), *dv = a.ptr<void>(9), *ws = a.ptr<void>(14);
    float *dg = a.ptr<float>(10), *dbeta = a.ptr<float>(11), *dw = a.ptr<float>(12);
    const natsl_params *p = a.params(13);
    const size_t wb = a.numel(14);
    NATSL_CALL(natsl_hybrid_bwd(q, k, vv, g, beta, route, dout, dq, dk, dv, dg, dbeta, dw, p, ws, wb, st));
}

PyObject *decode_step(PyObject *, PyObject *const *v, Py_ssize_t n) {
    if (!count_is(n, 13)) return nullptr;
    Args a{v};
    const void *q = a.ptr<void>(0), *k = a.ptr<void>(1), *vv = a.ptr<void>(2);
    const float *g = a.ptr<float>(3), *beta = a.ptr<float>(4);
    const uint8_t *route = a.ptr<uint8_t>(5);
    float *state = a.ptr<float>(6);
    void *kc = a.ptr<void>(7), *vc = a.ptr<void>(8), *out = a.ptr<void>(10), *ws = a.ptr<void>(12);
    int32_t *len = a.ptr<int32_t>(9);
    const int32_t cap = (int32_t)a.size(7, 2);
    const natsl_params *p = a.params(11);
    const size_t wb = a.numel(12);
    NATSL_CALL(natsl_decode_step(q, k, vv, g, beta, route, state, kc, vc, len, cap, out, p, ws, wb, st));
}

PyObject *decode_block_end(PyObject *, PyObject *const *v, Py_ssize_t n) {
    if (!count_is(n, 8)) return nullptr;
    Args a{v};
    const uint8_t *route = a.ptr<uint8_t>(0);
    const float *g = a.ptr<float>(1);
    float *state = a.ptr<float>(2), *start = a.ptr<float>(3);
    int32_t *len = a.ptr<int32_t>(4);
    const int32_t block_len = (int32_t)a.integer(5);
    const natsl_params *p = a.params(6);
    void *ws = a.ptr<void>(7);
    const size_t wb = a.numel(7);
    NATSL_CALL(natsl_decode_block_end(route, g, state, start, len, block_len, p, ws, wb, st));
}

PyObject *score_layer(PyObject *, PyObject *const *v, Py_ssize_t n) {
    if (!count_is(n, 5)) return nullptr;
    Args a{v};
    const void *x = a.ptr<void>(0);
    const float *w = a.ptr<float>(1);
    float *scores = a.ptr<float>(2);
    uint8_t *route = a.ptr<uint8_t>(3);
    const int32_t d_model = (int32_t)a.size(0, -1);
    const natsl_params *p = a.params(4);
    NATSL_CALL(natsl_score_layer(x, w, scores, route, d_model, p, st));
}

PyMethodDef kMethods[] = {
#define NATSL_DEF(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
    NATSL_DEF(hybrid_fwd), NATSL_DEF(hybrid_fwd_static), NATSL_DEF(hybrid_bwd), NATSL_DEF(decode_step),
    NATSL_DEF(decode_block_end), NATSL_DEF(score_layer), {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_natsl_py", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__natsl_py(void) { return PyModule_Create(&kModule); }
