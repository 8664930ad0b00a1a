// The Python binding's call path: tensors in, C ABI call out.  A ctypes call costs about 6 us of interpreter time for a layer
// pass (three attribute reads per tensor, a stream object, argument conversion) beside a kernel that takes 14; here the
// tensors are unpacked in C++, which leaves well under 1 us.  The module knows no symbol of the library: `init` hands over
// the entry points' addresses from the loaded libtaq.so.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <exception>

#include "taq.h"

namespace {

// The entry points, in the order of `NAMES`.
struct Entry {
    decltype(&taq_pack_weights) pack_weights;
    decltype(&taq_kv_project) kv_project;
    decltype(&taq_kv_project_a8) kv_project_a8;
    decltype(&taq_kv_project_batched) kv_project_batched;
    decltype(&taq_quantized_linear) quantized_linear;
    decltype(&taq_quantized_linear_i8) quantized_linear_i8;
    decltype(&taq_quantize_rows_f16) quantize_rows_f16;
    decltype(&taq_cross_attention) cross_attention;
    decltype(&taq_query_attention) query_attention;
    decltype(&taq_layer_forward) layer_forward;
    decltype(&taq_layer_forward_a8) layer_forward_a8;
    decltype(&taq_layer_forward_batched) layer_forward_batched;
    decltype(&taq_layer_forward_static) layer_forward_static;
} E;
const char* const NAMES[] = {"taq_pack_weights", "taq_kv_project", "taq_kv_project_a8", "taq_kv_project_batched", "taq_quantized_linear", "taq_quantized_linear_i8",
                             "taq_quantize_rows_f16", "taq_cross_attention", "taq_query_attention", "taq_layer_forward", "taq_layer_forward_a8",
                             "taq_layer_forward_batched", "taq_layer_forward_static"};
constexpr size_t N_ENTRY = sizeof(NAMES) / sizeof(NAMES[0]);
static_assert(sizeof(Entry) == N_ENTRY * sizeof(void*), "one address per name");

// The arguments of one call.  A conversion that fails sets the Python error and `bad`; the call is then not made.
struct Args {
    PyObject* const* v;
    bool bad = false;
    Args(PyObject* const* values, Py_ssize_t n, Py_ssize_t want) : v(values) {
        if (n != want) { PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, n); bad = true; }
    }
    void fail(PyObject* type, const char* what) { PyErr_SetString(type, what); bad = true; }
    template <typename T>
    const T* desc(int i) {                              // a ctypes structure
        Py_buffer b;
        if (bad) return nullptr;
        if (PyObject_GetBuffer(v[i], &b, PyBUF_SIMPLE) != 0) { bad = true; return nullptr; }
        const void* p = b.buf;
        const bool fits = b.len == (Py_ssize_t)sizeof(T);
        PyBuffer_Release(&b);                           // (the caller holds the object for the length of the call)
        if (!fits) { fail(PyExc_TypeError, "descriptor expected"); return nullptr; }
        return static_cast<const T*>(p);
    }
    const at::Tensor* tensor(int i) {
        if (bad || v[i] == Py_None) return nullptr;
        if (!THPVariable_Check(v[i])) { fail(PyExc_TypeError, "tensor expected"); return nullptr; }
        const at::Tensor& t = THPVariable_Unpack(v[i]);
        if (!t.is_cuda()) { fail(PyExc_TypeError, "device tensor expected"); return nullptr; }
        if (!t.is_contiguous()) { fail(PyExc_TypeError, "contiguous tensor expected"); return nullptr; }
        return &t;
    }
    void* ptr(int i) {
        const at::Tensor* t = tensor(i);
        if (!t) return nullptr;
        try {
            return t->data_ptr();
        } catch (const std::exception& e) {
            fail(PyExc_RuntimeError, e.what());
            return nullptr;
        }
    }
    size_t bytes(int i) { return bad || v[i] == Py_None ? 0 : (size_t)THPVariable_Unpack(v[i]).numel(); }     // (of a uint8 tensor)
    long long integer(int i) {
        if (bad) return 0;
        const long long x = PyLong_AsLongLong(v[i]);
        if (x == -1 && PyErr_Occurred()) bad = true;
        return x;
    }
    void* stream(int i) {                               // None (the current stream), an object with cuda_stream, or a handle
        if (bad) return nullptr;
        if (v[i] == Py_None) {
            try {
                return c10::cuda::getCurrentCUDAStream().stream();
            } catch (const std::exception& e) {
                fail(PyExc_RuntimeError, e.what());
                return nullptr;
            }
        }
        PyObject* h = PyObject_HasAttrString(v[i], "cuda_stream") ? PyObject_GetAttrString(v[i], "cuda_stream") : PyNumber_Long(v[i]);
        if (!h) { bad = true; return nullptr; }
        void* s = PyLong_AsVoidPtr(h);
        Py_DECREF(h);
        if (!s && PyErr_Occurred()) bad = true;
        return s;
    }
};

template <typename F>
PyObject* answer(const Args& a, F call) {
    if (a.bad) return nullptr;
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = (int)call();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

#define TAQ_FN(name) PyObject* name(PyObject*, PyObject* const* v, Py_ssize_t n)

TAQ_FN(pack_weights) {                                  // desc, W, bias, packed, stream
    Args a(v, n, 5);
    auto d = a.desc<taq_weight_desc>(0);
    auto W = (const float*)a.ptr(1), b = (const float*)a.ptr(2);
    void *p = a.ptr(3), *s = a.stream(4);
    const size_t nb = a.bytes(3);
    return answer(a, [&] { return E.pack_weights(d, W, b, p, nb, s); });
}
TAQ_FN(kv_project) {                                    // desc, ctx, Wk, Wv, mask, kv, stream
    Args a(v, n, 7);
    auto d = a.desc<taq_layer_desc>(0);
    void *x = a.ptr(1), *k = a.ptr(2), *w = a.ptr(3), *m = a.ptr(4), *kv = a.ptr(5), *s = a.stream(6);
    const size_t nb = a.bytes(5);
    return answer(a, [&] { return E.kv_project(d, x, k, w, (const uint8_t*)m, kv, nb, s); });
}
TAQ_FN(kv_project_a8) {                                 // desc, ctx, Wk, Wv, mask, kv, workspace, stream
    Args a(v, n, 8);
    auto d = a.desc<taq_layer_desc>(0);
    void *x = a.ptr(1), *k = a.ptr(2), *w = a.ptr(3), *m = a.ptr(4), *kv = a.ptr(5), *ws = a.ptr(6), *s = a.stream(7);
    const size_t nb = a.bytes(5), wb = a.bytes(6);
    return answer(a, [&] { return E.kv_project_a8(d, x, k, w, (const uint8_t*)m, kv, nb, ws, wb, s); });
}
TAQ_FN(kv_project_batched) {                            // desc, reqs, n_requests, ctx, stream
    Args a(v, n, 5);
    auto d = a.desc<taq_layer_desc>(0);
    auto r = (const taq_request*)a.ptr(1);
    const int32_t nr = (int32_t)a.integer(2);
    void *x = a.ptr(3), *s = a.stream(4);
    return answer(a, [&] { return E.kv_project_batched(d, r, nr, x, s); });
}
TAQ_FN(quantized_linear) {                              // desc, x, rows, W, y, out_kind, heads, scales, stream
    Args a(v, n, 9);
    auto d = a.desc<taq_weight_desc>(0);
    void *x = a.ptr(1), *W = a.ptr(3), *y = a.ptr(4), *sc = a.ptr(7), *s = a.stream(8);
    const long long rows = a.integer(2), kind = a.integer(5), heads = a.integer(6);
    return answer(a, [&] { return E.quantized_linear(d, x, rows, W, y, (int32_t)kind, (int32_t)heads, (float*)sc, s); });
}
TAQ_FN(quantized_linear_i8) {                           // desc, codes, x_scales, rows, W, y, out_kind, heads, scales, stream
    Args a(v, n, 10);
    auto d = a.desc<taq_weight_desc>(0);
    void *x = a.ptr(1), *xs = a.ptr(2), *W = a.ptr(4), *y = a.ptr(5), *sc = a.ptr(8), *s = a.stream(9);
    const long long rows = a.integer(3), kind = a.integer(6), heads = a.integer(7);
    return answer(a, [&] { return E.quantized_linear_i8(d, (const int8_t*)x, (const float*)xs, rows, W, y, (int32_t)kind, (int32_t)heads, (float*)sc, s); });
}
TAQ_FN(quantize_rows_f16) {                             // x, rows, cols, codes, scales, stream
    Args a(v, n, 6);
    void *x = a.ptr(0), *c = a.ptr(3), *sc = a.ptr(4), *s = a.stream(5);
    const long long rows = a.integer(1), cols = a.integer(2);
    return answer(a, [&] { return E.quantize_rows_f16(x, rows, (int32_t)cols, (int8_t*)c, (float*)sc, s); });
}
TAQ_FN(cross_attention) {                               // desc, q, q_scales, kv, mask, o, stream
    Args a(v, n, 7);
    auto d = a.desc<taq_layer_desc>(0);
    void *q = a.ptr(1), *qs = a.ptr(2), *kv = a.ptr(3), *m = a.ptr(4), *o = a.ptr(5), *s = a.stream(6);
    return answer(a, [&] { return E.cross_attention(d, q, (const float*)qs, kv, (const uint8_t*)m, o, s); });
}
TAQ_FN(query_attention) {                               // desc, x, Wq, kv, mask, o, workspace, stream
    Args a(v, n, 8);
    auto d = a.desc<taq_layer_desc>(0);
    void *x = a.ptr(1), *W = a.ptr(2), *kv = a.ptr(3), *m = a.ptr(4), *o = a.ptr(5), *ws = a.ptr(6), *s = a.stream(7);
    const size_t wb = a.bytes(6);
    return answer(a, [&] { return E.query_attention(d, x, W, kv, (const uint8_t*)m, o, ws, wb, s); });
}
template <typename F>
PyObject* layer(F Entry::*fn, PyObject* const* v, Py_ssize_t n) {      // desc, x, Wq, Wout, kv, mask, y, workspace, stream
    Args a(v, n, 9);
    auto d = a.desc<taq_layer_desc>(0);
    void *x = a.ptr(1), *q = a.ptr(2), *o = a.ptr(3), *kv = a.ptr(4), *m = a.ptr(5), *y = a.ptr(6), *ws = a.ptr(7), *s = a.stream(8);
    const size_t wb = a.bytes(7);
    return answer(a, [&] { return (E.*fn)(d, x, q, o, kv, (const uint8_t*)m, y, ws, wb, s); });
}
TAQ_FN(layer_forward) { return layer(&Entry::layer_forward, v, n); }
TAQ_FN(layer_forward_a8) { return layer(&Entry::layer_forward_a8, v, n); }
TAQ_FN(layer_forward_batched) {                         // desc, reqs, n_requests, x, y, workspace, stream
    Args a(v, n, 7);
    auto d = a.desc<taq_layer_desc>(0);
    auto r = (const taq_request*)a.ptr(1);
    const int32_t nr = (int32_t)a.integer(2);
    void *x = a.ptr(3), *y = a.ptr(4), *ws = a.ptr(5), *s = a.stream(6);
    const size_t wb = a.bytes(5);
    return answer(a, [&] { return E.layer_forward_batched(d, r, nr, x, y, ws, wb, s); });
}
TAQ_FN(layer_forward_static) {                          // desc, x, Wq, Wout, kv, mask, y, stream
    Args a(v, n, 8);
    auto d = a.desc<taq_layer_desc>(0);
    void *x = a.ptr(1), *q = a.ptr(2), *o = a.ptr(3), *kv = a.ptr(4), *m = a.ptr(5), *y = a.ptr(6), *s = a.stream(7);
    return answer(a, [&] { return E.layer_forward_static(d, x, q, o, kv, (const uint8_t*)m, y, s); });
}

PyObject* init(PyObject*, PyObject* const* v, Py_ssize_t n) {          // the addresses of NAMES
    if (n != (Py_ssize_t)N_ENTRY) { PyErr_SetString(PyExc_TypeError, "one address per entry point expected"); return nullptr; }
    void* p[N_ENTRY];
    for (size_t i = 0; i < N_ENTRY; ++i) {
        p[i] = PyLong_AsVoidPtr(v[i]);
        if (!p[i]) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null entry point"); return nullptr; }
    }
    memcpy(&E, p, sizeof(p));
    Py_RETURN_NONE;
}
PyObject* names(PyObject*, PyObject*) {
    PyObject* t = PyTuple_New(N_ENTRY);
    for (size_t i = 0; t && i < N_ENTRY; ++i) PyTuple_SET_ITEM(t, i, PyUnicode_FromString(NAMES[i]));
    return t;
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef METHODS[] = {FAST(init), {"names", names, METH_NOARGS, nullptr}, FAST(pack_weights), FAST(kv_project), FAST(kv_project_a8), FAST(kv_project_batched),
                         FAST(quantized_linear), FAST(quantized_linear_i8), FAST(quantize_rows_f16), FAST(cross_attention), FAST(query_attention), FAST(layer_forward),
                         FAST(layer_forward_a8), FAST(layer_forward_batched), FAST(layer_forward_static), {nullptr, nullptr, 0, nullptr}};
PyModuleDef MODULE = {PyModuleDef_HEAD_INIT, "_taq_call", nullptr, -1, METHODS, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__taq_call(void) { return PyModule_Create(&MODULE); }
