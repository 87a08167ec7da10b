// The linears' Python calls: tensors are checked and taken apart here and the library is called with their addresses.
//
// What bounds it.  Nothing but the host: a decode step is a chain of calls whose kernels take 7 to 20 us each, and taking ten tensors and
// numbers apart in Python and ctypes took 6 us of the 10 us between two calls, so that a layer of four 4-bit linears at one row took 41 us
// however fast its kernels were.  Now 3 to 4.5 us between two calls (2.5 to 4 of them the library's, most of it the launch), and those four linears take
// 38.7 us, which is what their kernels take.
//
// Each function returns the library's status, or -1 for arguments that it does not take; the caller then finds out in Python what is wrong with them.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "dmr.h"

namespace {

decltype(&dmr_lowbit_linear) g_lowbit = nullptr;
decltype(&dmr_dense_linear) g_dense = nullptr;
decltype(&dmr_routed_linear) g_routed = nullptr;

const at::Tensor *tensor(PyObject *o) { return THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr; }

// A contiguous tensor on a GPU, of the given type and, if it is not negative, number of dimensions.
const at::Tensor *device_tensor(PyObject *o, at::ScalarType type, int dims = -1) {
    const at::Tensor *t = tensor(o);
    return t && t->is_cuda() && t->scalar_type() == type && (dims < 0 || t->dim() == dims) && t->is_contiguous() ? t : nullptr;
}

// Addresses of tensors; false where one is missing.
bool addresses(std::initializer_list<const at::Tensor *> tensors, void **out) {
    for (const at::Tensor *t : tensors) {
        if (!t) return false;
        *out++ = t->data_ptr();
    }
    return true;
}

// The stream a call is enqueued on: the given handle, or (None) the current one.
bool stream_of(PyObject *o, void **stream) {
    if (o == Py_None) {
        *stream = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    *stream = PyLong_AsVoidPtr(o);
    return !PyErr_Occurred();
}

bool ints(PyObject *const *args, int n, int *out) {
    for (int i = 0; i < n; ++i) {
        const long v = PyLong_AsLong(args[i]);
        if (v == -1 && PyErr_Occurred()) return false;
        if (v < INT32_MIN || v > INT32_MAX) return false;
        out[i] = (int)v;
    }
    return true;
}

PyObject *refused() {
    PyErr_Clear();
    return PyLong_FromLong(-1);
}

// A tensor that cannot say its size, order or address (compressed sparse, symbolic or jagged sizes, no storage) throws when it is asked.
template <PyObject *take(PyObject *const *, Py_ssize_t)>
PyObject *guarded(PyObject *, PyObject *const *args, Py_ssize_t n) {
    try {
        return take(args, n);
    } catch (const std::exception &) {
        return refused();
    }
}

template <class F>
PyObject *call(F f) noexcept {  // other Python threads run meanwhile
    int r;
    Py_BEGIN_ALLOW_THREADS
    r = (int)f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(r);
}

// bind(lowbit, dense, routed): addresses of the library's functions
PyObject *bind(PyObject *, PyObject *const *args, Py_ssize_t n) {
    if (n != 3) return refused();
    g_lowbit = reinterpret_cast<decltype(g_lowbit)>(PyLong_AsVoidPtr(args[0]));
    g_dense = reinterpret_cast<decltype(g_dense)>(PyLong_AsVoidPtr(args[1]));
    g_routed = reinterpret_cast<decltype(g_routed)>(PyLong_AsVoidPtr(args[2]));
    if (PyErr_Occurred()) return nullptr;
    Py_RETURN_NONE;
}

at::ScalarType out_type(int out) { return out == DMR_OUT_F32 ? at::kFloat : at::kBFloat16; }

// lowbit(X, qweight, scales, zeros, N, K, bits, group, Y, out, workspace, stream)
PyObject *lowbit(PyObject *const *args, Py_ssize_t n) {
    if (n != 12 || !g_lowbit) return refused();
    const at::Tensor *X = device_tensor(args[0], at::kBFloat16, 2), *ws = tensor(args[10]);
    int v[4], out;
    void *stream, *p[6];
    if (!X || !ints(args + 4, 4, v) || !ints(args + 9, 1, &out) || X->size(1) != v[1]) return refused();
    if (!addresses({X, tensor(args[1]), tensor(args[2]), tensor(args[3]), device_tensor(args[8], out_type(out)), ws}, p) || !stream_of(args[11], &stream)) return refused();
    const int M = (int)X->size(0);
    const size_t ws_bytes = (size_t)ws->numel();
    const dmr_qformat_t f = {v[2], v[3]};
    return call([&] { return g_lowbit(p[0], M, p[1], p[2], p[3], v[0], v[1], f, p[4], (dmr_out_t)out, p[5], ws_bytes, stream); });
}

// dense(X, W, Y, out, workspace, stream)
PyObject *dense(PyObject *const *args, Py_ssize_t n) {
    if (n != 6 || !g_dense) return refused();
    const at::Tensor *X = device_tensor(args[0], at::kBFloat16, 2), *W = device_tensor(args[1], at::kBFloat16, 2), *ws = tensor(args[4]);
    int out;
    void *stream, *p[4];
    if (!X || !W || !ints(args + 3, 1, &out) || X->size(1) != W->size(1)) return refused();
    if (!addresses({X, W, device_tensor(args[2], out_type(out)), ws}, p) || !stream_of(args[5], &stream)) return refused();
    const int M = (int)X->size(0), N = (int)W->size(0), K = (int)W->size(1);
    const size_t ws_bytes = (size_t)ws->numel();
    return call([&] { return g_dense(p[0], M, p[1], N, K, p[2], (dmr_out_t)out, p[3], ws_bytes, stream); });
}

// routed(X, mask, W, qweight, scales, zeros, N, K, bits, group, Y, out, workspace, stream)
PyObject *routed(PyObject *const *args, Py_ssize_t n) {
    if (n != 14 || !g_routed) return refused();
    const at::Tensor *X = device_tensor(args[0], at::kBFloat16, 2), *mask = device_tensor(args[1], at::kByte), *W = device_tensor(args[2], at::kBFloat16, 2);
    const at::Tensor *ws = tensor(args[12]);
    int v[4], out;
    void *stream, *p[8];
    if (!X || !mask || !W || !ints(args + 6, 4, v) || !ints(args + 11, 1, &out)) return refused();
    if (mask->numel() != X->size(0) || W->size(0) != v[0] || W->size(1) != v[1] || X->size(1) != v[1]) return refused();
    if (!addresses({X, mask, W, tensor(args[3]), tensor(args[4]), tensor(args[5]), device_tensor(args[10], out_type(out)), ws}, p) || !stream_of(args[13], &stream))
        return refused();
    const int M = (int)X->size(0);
    const size_t ws_bytes = (size_t)ws->numel();
    const dmr_qformat_t f = {v[2], v[3]};
    return call([&] {
        return g_routed(p[0], M, (const uint8_t *)p[1], p[2], p[3], p[4], p[5], v[0], v[1], f, p[6], (dmr_out_t)out, p[7], ws_bytes, stream);
    });
}

PyMethodDef g_methods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(bind)), METH_FASTCALL, nullptr},
    {"lowbit", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<lowbit>)), METH_FASTCALL, nullptr},
    {"dense", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<dense>)), METH_FASTCALL, nullptr},
    {"routed", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<routed>)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() { return PyModule_Create(&g_module); }
