// CPython entry to the fused calls: takes the torch tensors as they are and calls the C ABI.
//
// What bounds a short call is the host: with thirteen arguments marshalled through ctypes, and a method call or two on every
// tensor, calls on a 4096 x 4096 layer followed each other every 10.8 us although the kernel runs 5; here a tensor
// costs a type check and a pointer read, and they follow every 5.1 us.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "fq.h"

namespace {

// What a call of the tensor library threw (a tensor without storage, or of a kind that has no strides) as a Python error: nothing
// may leave a C entry.
template <class F>
bool guarded(F&& f) {
    try {
        return f();
    } catch (const c10::Error& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return false;
}

// Device pointer of a contiguous CUDA tensor; None is the null pointer.  `written`: the call writes to it, so that a
// tensor that shares its storage until it is written gets one of its own.  `bytes` (if given): its size.
bool device_pointer(PyObject* o, void** out, bool written = false, size_t* bytes = nullptr) {
    if (bytes) *bytes = 0;
    if (o == Py_None) {
        *out = nullptr;
        return true;
    }
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a torch tensor");
        return false;
    }
    return guarded([&] {
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda() || !t.is_contiguous()) {
            PyErr_SetString(PyExc_ValueError, "expected a contiguous CUDA tensor");
            return false;
        }
        *out = written ? t.mutable_data_ptr() : const_cast<void*>(t.const_data_ptr());
        if (bytes) *bytes = t.nbytes();
        return true;
    });
}

// The stream's handle: the given stream object's, or the current stream of the current device.
bool stream_handle(PyObject* o, void** out) {
    if (o == Py_None)                                      // (throws where there is no usable device)
        return guarded([&] {
            *out = c10::cuda::getCurrentCUDAStream().stream();
            return true;
        });
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) return false;
    *out = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
}

bool host_pointer(PyObject* o, void** out) {
    *out = PyLong_AsVoidPtr(o);
    return !PyErr_Occurred();
}

struct LayoutView {
    Py_buffer b{};
    bool held = false;
    ~LayoutView() { if (held) PyBuffer_Release(&b); }
    const fq_layout_t* get(PyObject* o) {
        if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return nullptr;
        held = true;
        if ((size_t)b.len != sizeof(fq_layout_t)) {
            PyErr_SetString(PyExc_TypeError, "expected a Layout");
            return nullptr;
        }
        return (const fq_layout_t*)b.buf;
    }
};

bool take(PyObject* const* args, Py_ssize_t n, Py_ssize_t want) {
    if (n != want) PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return n == want;
}

// L, X, M, wq, scale, zero, tile_indptr, bucket_info, packed, Y, workspace, stream -> status
PyObject* fused(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!take(a, n, 12)) return nullptr;
    LayoutView lv;
    const fq_layout_t* L = lv.get(a[0]);
    if (!L) return nullptr;
    const unsigned long M = PyLong_AsUnsignedLongMask(a[2]);
    if (PyErr_Occurred()) return nullptr;
    void *X, *w[6], *Y, *ws, *stream;
    if (!device_pointer(a[1], &X)) return nullptr;
    for (int i = 0; i < 6; ++i)
        if (!device_pointer(a[3 + i], &w[i])) return nullptr;
    size_t ws_bytes;
    if (!device_pointer(a[9], &Y, true) || !device_pointer(a[10], &ws, true, &ws_bytes) || !stream_handle(a[11], &stream)) return nullptr;
    fq_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = fq_fused_w4a16_outlier_gemm(L, X, (uint32_t)M, w[0], w[1], w[2], w[3], w[4], w[5], Y, ws, ws_bytes, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

// L, X_host, M, x_dev, wq, scale, zero, tile_indptr, bucket_info, packed, y_dev, Y_host, workspace, stream, wait -> status
PyObject* host_io(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!take(a, n, 15)) return nullptr;
    LayoutView lv;
    const fq_layout_t* L = lv.get(a[0]);
    if (!L) return nullptr;
    const unsigned long M = PyLong_AsUnsignedLongMask(a[2]);
    if (PyErr_Occurred()) return nullptr;
    void *xh, *yh, *x, *w[6], *y, *ws, *stream;
    if (!host_pointer(a[1], &xh) || !host_pointer(a[11], &yh) || !device_pointer(a[3], &x, true)) return nullptr;
    for (int i = 0; i < 6; ++i)
        if (!device_pointer(a[4 + i], &w[i])) return nullptr;
    size_t ws_bytes;
    if (!device_pointer(a[10], &y, true) || !device_pointer(a[12], &ws, true, &ws_bytes) || !stream_handle(a[13], &stream)) return nullptr;
    const auto call = a[14] == Py_True ? fq_fused_host_io : fq_fused_host_io_async;
    fq_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = call(L, xh, (uint32_t)M, x, w[0], w[1], w[2], w[3], w[4], w[5], y, yh, ws, ws_bytes, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

PyMethodDef methods[] = {
    {"fused", (PyCFunction)(void (*)(void))fused, METH_FASTCALL, nullptr},
    {"host_io", (PyCFunction)(void (*)(void))host_io, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fqcall", nullptr, -1, methods};

}  // namespace

// `built_for`: the torch whose C++ interface this file was compiled against.
PyMODINIT_FUNC PyInit__fqcall(void) {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", FQ_TORCH_TAG) != 0) Py_CLEAR(m);
    return m;
}
