// The per-call half of the Python binding, as a CPython extension: what binding.py does between a caller's tensors and
// the C ABI for the two calls that a decode loop makes per layer (one linear layer, one layer set).
//
// One token through a 4096 x 4096 layer takes 5.7 us on the device.  Checked and marshalled in Python (six tensors, a
// numpy bit map, the stream, an output, a ctypes call of thirteen arguments) the call took 15 us of the host, so the
// device waited for it; here the tensors are read without the interpreter, and the calls of a loop follow each other every
// 6.0 us (10.2 instead of 16.4 at a group size of 64).  A layer's very first call: 37 -> 24 us.
//
// Nothing is decided here.  A call that is not the plain one (another dtype or layout, a tensor subclass, a bit map that
// is not a one-dimensional uint8 buffer, ...) returns None before anything has been enqueued and binding.py takes its
// general path, which converts or raises.  The entry points of the C ABI arrive as addresses, so this file links
// against nothing of the CUDA library and keeps no state.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

using LinearFn = int (*)(const void*, const void*, const uint8_t*, const void*, const void*, void*, int, int, int, int, void*, size_t, void*);
using SetFn = int (*)(const void*, const void*, void*, size_t, void*);

const at::Tensor* plain(PyObject* o, c10::ScalarType dtype) {
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    return t.is_cuda() && t.layout() == c10::kStrided && t.scalar_type() == dtype && t.is_contiguous() ? &t : nullptr;
}

bool as_int(PyObject* o, int* out) {
    if (!PyLong_CheckExact(o)) return false;
    int overflow = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &overflow);
    if (overflow != 0 || v < INT_MIN || v > INT_MAX) return false;
    *out = static_cast<int>(v);
    return true;
}

void* stream_of(const at::Tensor& t) { return c10::cuda::getCurrentCUDAStream(t.get_device()).stream(); }

// The bit map of a layer: a one-dimensional uint8 array that numpy can be asked for without a copy.
struct Bits {
    Py_buffer b;
    bool held = false;
    bool open(PyObject* o) {
        if (PyBytes_Check(o) || PyByteArray_Check(o) || PyMemoryView_Check(o)) return false;      // the general path says what they are
        if (PyObject_GetBuffer(o, &b, PyBUF_FORMAT | PyBUF_ND | PyBUF_C_CONTIGUOUS) != 0) { PyErr_Clear(); return false; }
        held = true;
        return b.ndim == 1 && b.itemsize == 1 && b.format != nullptr && b.format[0] == 'B' && b.format[1] == 0;
    }
    ~Bits() { if (held) PyBuffer_Release(&b); }
};

// What torch throws (a tensor without storage or of a layout that has no strides, no memory left) leaves as the Python
// exception that the same call in Python raises.
// linear(address, x, packed, bits, scales, zeros, N, workspace, out or None, g) -> y, or the status of a call that failed, or None (see above)
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 10) { PyErr_SetString(PyExc_TypeError, "linear: 10 arguments"); return nullptr; }
    LinearFn fn = reinterpret_cast<LinearFn>(PyLong_AsVoidPtr(a[0]));
    if (fn == nullptr) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "linear: no entry point"); return nullptr; }
    int N = 0, g = 0;
    const at::Tensor *x = plain(a[1], at::kHalf), *packed = plain(a[2], at::kByte), *scales = plain(a[4], at::kHalf),
                     *zeros = plain(a[5], at::kHalf), *ws = plain(a[7], at::kByte);
    if (x == nullptr || packed == nullptr || scales == nullptr || zeros == nullptr || ws == nullptr || x->dim() != 2 ||
        !as_int(a[6], &N) || N < 0 || !as_int(a[9], &g) || x->size(0) > INT_MAX || x->size(1) > INT_MAX)
        Py_RETURN_NONE;
    const at::Tensor* given = nullptr;
    if (a[8] != Py_None && (given = plain(a[8], at::kHalf)) == nullptr) Py_RETURN_NONE;
    Bits bits;
    if (!bits.open(a[3])) Py_RETURN_NONE;
    const int M = static_cast<int>(x->size(0)), K = static_cast<int>(x->size(1));
    at::Tensor fresh;
    if (given == nullptr) fresh = at::empty({M, N}, x->options());
    const at::Tensor& y = given != nullptr ? *given : fresh;
    void *xp = x->data_ptr(), *wp = packed->data_ptr(), *sp = scales->data_ptr(), *zp = zeros->data_ptr(), *yp = y.data_ptr();
    void *wsp = ws->data_ptr(), *stream = stream_of(*x);
    const size_t wsb = static_cast<size_t>(ws->numel());
    int status = 0;
    Py_BEGIN_ALLOW_THREADS                      // the tensors and the bit map are held by the caller's arguments
    status = fn(xp, wp, static_cast<const uint8_t*>(bits.b.buf), sp, zp, yp, M, N, K, g, wsp, wsb, stream);
    Py_END_ALLOW_THREADS
    if (status != 0) return PyLong_FromLong(status);
    return given != nullptr ? Py_NewRef(a[8]) : THPVariable_Wrap(fresh);
    END_HANDLE_TH_ERRORS
}

// run_set(address, launch record, plan, workspace) -> status, or None
PyObject* run_set(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 4) { PyErr_SetString(PyExc_TypeError, "run_set: 4 arguments"); return nullptr; }
    SetFn fn = reinterpret_cast<SetFn>(PyLong_AsVoidPtr(a[0]));
    const void* info = fn != nullptr ? PyLong_AsVoidPtr(a[1]) : nullptr;
    if (fn == nullptr || info == nullptr) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "run_set: no entry point"); return nullptr; }
    const at::Tensor *plan = plain(a[2], at::kByte), *ws = plain(a[3], at::kByte);
    if (plan == nullptr || ws == nullptr) Py_RETURN_NONE;
    void *pp = plan->data_ptr(), *wp = ws->data_ptr(), *stream = stream_of(*plan);
    const size_t wsb = static_cast<size_t>(ws->numel());
    int status = 0;
    Py_BEGIN_ALLOW_THREADS
    status = fn(info, pp, wp, wsb, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"linear", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(linear)), METH_FASTCALL, nullptr},
    {"run_set", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(run_set)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "slim_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_slim_host(void) { return PyModule_Create(&module_def); }
