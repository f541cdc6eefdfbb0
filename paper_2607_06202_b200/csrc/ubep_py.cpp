// CPython module for the calls a layer makes every step: tensors and the current stream to the C ABI of
// libubep.so without going through ctypes.
//
// Why it exists: on a B200 host a decode-sized layer takes the GPU 8 to 25 us, and through ctypes the two
// calls took the host 20.4 us -- 3.6 us per call to ask torch for the current stream object, 0.2 us per
// pointer, 0.6 us for ctypes itself, 2.5 us for torch.empty -- against 2.6 to 2.9 us per kernel launch,
// which is what is left.  Nothing here is cached between calls.
//
// The library's entry points are handed over by address (bind), so this module links neither libubep.so
// nor the CUDA runtime.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <exception>

#include "../../include/ubep.h"

namespace {

decltype(&ubep_dispatch) f_dispatch;
decltype(&ubep_combine) f_combine;
decltype(&ubep_get_dispatch_layout) f_layout;
decltype(&ubep_dispatch_sync) f_dispatch_sync;

// An argument that must be a contiguous tensor, or None where the C ABI takes a null pointer.
bool tensor_arg(PyObject* o, void** ptr, const at::Tensor** t = nullptr) {
    if (o == Py_None) {
        *ptr = nullptr;
        return true;
    }
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "expected a tensor or None, got %s", Py_TYPE(o)->tp_name);
        return false;
    }
    const at::Tensor& v = THPVariable_Unpack(o);
    if (!v.is_contiguous()) {
        PyErr_SetString(PyExc_AssertionError, "tensor is not contiguous");
        return false;
    }
    *ptr = v.data_ptr();
    if (t) *t = &v;
    return true;
}

bool rows_of(PyObject* o, int32_t* rows) {   // first dimension of a tensor
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "expected a tensor, got %s", Py_TYPE(o)->tp_name);
        return false;
    }
    const at::Tensor& v = THPVariable_Unpack(o);
    if (v.dim() < 1) {
        PyErr_SetString(PyExc_IndexError, "tensor has no dimension");
        return false;
    }
    const int64_t n = v.size(0);
    *rows = n > INT32_MAX ? INT32_MAX : (int32_t)n;
    return true;
}

bool int_arg(PyObject* o, long long* v) {
    *v = PyLong_AsLongLong(o);
    return !(*v == -1 && PyErr_Occurred());
}

bool count_arg(PyObject* o, int32_t* v) {   // an int32 of the C ABI (out of range: an argument error there)
    long long n;
    if (!int_arg(o, &n)) return false;
    *v = n < INT32_MIN || n > INT32_MAX ? -1 : (int32_t)n;
    return true;
}

// The library's buffer handle as an integer; None after the buffer was closed.
bool handle_arg(PyObject* o, ubep_buffer_t** buf) {
    *buf = o == Py_None ? nullptr : static_cast<ubep_buffer_t*>(PyLong_AsVoidPtr(o));
    return !PyErr_Occurred();
}

// None = torch's current stream; otherwise an object with a `cuda_stream` handle, or the handle as anything int() takes.
bool stream_arg(PyObject* o, void** st) {
    if (o == Py_None) {
        *st = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* h = nullptr;
    if (PyLong_Check(o)) {
        h = Py_NewRef(o);
    } else if (PyObject_HasAttrString(o, "cuda_stream")) {
        h = PyObject_GetAttrString(o, "cuda_stream");
    } else {
        h = PyNumber_Long(o);
    }
    if (!h) return false;
    *st = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
}

bool want_args(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return false;
}

PyObject* translate_exception() {
    try {
        throw;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}

// The GIL is released around a library call, as ctypes does: a launch may wait for room in the stream's queue.
template <typename F>
int without_gil(F call) {
    PyThreadState* state = PyEval_SaveThread();
    const int rc = call();
    PyEval_RestoreThread(state);
    return rc;
}

// Every call below returns an int (the C ABI's code) or, where it makes its outputs, those.

// dispatch(handle, x, topk_idx, topk_w, T or None, stream): T defaults to x's rows
PyObject* py_dispatch(PyObject*, PyObject* const* a, Py_ssize_t n) {
    try {
        if (!want_args(n, 6)) return nullptr;
        ubep_buffer_t* buf;
        void *x, *idx, *w, *st;
        int32_t T = 0;
        if (!handle_arg(a[0], &buf) || !tensor_arg(a[1], &x) || !tensor_arg(a[2], &idx) || !tensor_arg(a[3], &w) ||
            !(a[4] == Py_None ? rows_of(a[1], &T) : count_arg(a[4], &T)) || !stream_arg(a[5], &st))
            return nullptr;
        return PyLong_FromLong(without_gil([&] {
            return f_dispatch(buf, x, static_cast<const int32_t*>(idx), static_cast<const float*>(w), T, st);
        }));
    } catch (...) {
        return translate_exception();
    }
}

// dispatch_sync(handle, protocol, x, topk_idx, topk_w, T or None, stream)
PyObject* py_dispatch_sync(PyObject*, PyObject* const* a, Py_ssize_t n) {
    try {
        if (!want_args(n, 7)) return nullptr;
        ubep_buffer_t* buf;
        void *x, *idx, *w, *st;
        int32_t T = 0, proto;
        if (!handle_arg(a[0], &buf) || !count_arg(a[1], &proto) || !tensor_arg(a[2], &x) || !tensor_arg(a[3], &idx) ||
            !tensor_arg(a[4], &w) || !(a[5] == Py_None ? rows_of(a[2], &T) : count_arg(a[5], &T)) ||
            !stream_arg(a[6], &st))
            return nullptr;
        return PyLong_FromLong(without_gil([&] {
            return f_dispatch_sync(buf, proto, x, static_cast<const int32_t*>(idx), static_cast<const float*>(w), T, st);
        }));
    } catch (...) {
        return translate_exception();
    }
}

// combine(handle, y, topk_w, T or None, out, stream): T defaults to topk_w's rows; the code
PyObject* py_combine(PyObject*, PyObject* const* a, Py_ssize_t n) {
    try {
        if (!want_args(n, 6)) return nullptr;
        ubep_buffer_t* buf;
        void *y, *w, *out, *st;
        int32_t T = 0;
        if (!handle_arg(a[0], &buf) || !tensor_arg(a[1], &y) || !tensor_arg(a[2], &w) ||
            !(a[3] == Py_None ? rows_of(a[2], &T) : count_arg(a[3], &T)) || !tensor_arg(a[4], &out) ||
            !stream_arg(a[5], &st))
            return nullptr;
        return PyLong_FromLong(without_gil([&] {
            return f_combine(buf, y, static_cast<const float*>(w), T, out, st);
        }));
    } catch (...) {
        return translate_exception();
    }
}

// combine_new(handle, y, topk_w, hidden, device, stream): the bf16 output [rows of topk_w, hidden], or the code
PyObject* py_combine_new(PyObject*, PyObject* const* a, Py_ssize_t n) {
    try {
        if (!want_args(n, 6)) return nullptr;
        ubep_buffer_t* buf;
        void *y, *w, *st;
        int32_t T;
        long long hidden, device;
        if (!handle_arg(a[0], &buf) || !tensor_arg(a[1], &y) || !tensor_arg(a[2], &w) || !rows_of(a[2], &T) ||
            !int_arg(a[3], &hidden) || !int_arg(a[4], &device) || !stream_arg(a[5], &st))
            return nullptr;
        at::Tensor out = at::detail::empty_cuda({(int64_t)T, (int64_t)hidden}, at::kBFloat16,
                                                c10::Device(c10::kCUDA, (c10::DeviceIndex)device), c10::nullopt);
        void* po = out.data_ptr();
        const int rc = without_gil([&] { return f_combine(buf, y, static_cast<const float*>(w), T, po, st); });
        if (rc != UBEP_OK) return PyLong_FromLong(rc);
        return THPVariable_Wrap(std::move(out));
    } catch (...) {
        return translate_exception();
    }
}

// layout(handle, topk_idx, T, tokens_per_rank, tokens_per_expert, is_token_in_rank, stream): the code
PyObject* py_layout(PyObject*, PyObject* const* a, Py_ssize_t n) {
    try {
        if (!want_args(n, 7)) return nullptr;
        ubep_buffer_t* buf;
        void *idx, *npr, *npe, *itr, *st;
        int32_t T;
        if (!handle_arg(a[0], &buf) || !tensor_arg(a[1], &idx) || !count_arg(a[2], &T) || !tensor_arg(a[3], &npr) ||
            !tensor_arg(a[4], &npe) || !tensor_arg(a[5], &itr) || !stream_arg(a[6], &st))
            return nullptr;
        return PyLong_FromLong(without_gil([&] {
            return f_layout(buf, static_cast<const int32_t*>(idx), T, static_cast<int32_t*>(npr),
                            static_cast<int32_t*>(npe), static_cast<uint8_t*>(itr), st);
        }));
    } catch (...) {
        return translate_exception();
    }
}

// layout_new(handle, topk_idx, num_ranks, num_experts, device, stream): the tuple (tokens_per_rank [R] int32,
// tokens_per_expert [E] int32, is_token_in_rank [T, R] uint8), or the code.  Three allocations: each result is a tensor of
// its own, which a caller may keep, save or resize without the others.
PyObject* py_layout_new(PyObject*, PyObject* const* a, Py_ssize_t n) {
    try {
        if (!want_args(n, 6)) return nullptr;
        ubep_buffer_t* buf;
        void *idx, *st;
        int32_t T;
        long long R, E, device;
        if (!handle_arg(a[0], &buf) || !tensor_arg(a[1], &idx) || !rows_of(a[1], &T) || !int_arg(a[2], &R) ||
            !int_arg(a[3], &E) || !int_arg(a[4], &device) || !stream_arg(a[5], &st))
            return nullptr;
        const c10::Device dev(c10::kCUDA, (c10::DeviceIndex)device);
        at::Tensor parts[3] = {at::detail::empty_cuda({(int64_t)R}, at::kInt, dev, c10::nullopt),
                               at::detail::empty_cuda({(int64_t)E}, at::kInt, dev, c10::nullopt),
                               at::detail::empty_cuda({(int64_t)T, (int64_t)R}, at::kByte, dev, c10::nullopt)};
        void* po[3] = {parts[0].data_ptr(), parts[1].data_ptr(), parts[2].data_ptr()};
        const int rc = without_gil([&] {
            return f_layout(buf, static_cast<const int32_t*>(idx), T, static_cast<int32_t*>(po[0]),
                            static_cast<int32_t*>(po[1]), static_cast<uint8_t*>(po[2]), st);
        });
        if (rc != UBEP_OK) return PyLong_FromLong(rc);
        PyObject* out = PyTuple_New(3);
        if (!out) return nullptr;
        for (int i = 0; i < 3; ++i) {
            PyObject* o = THPVariable_Wrap(std::move(parts[i]));
            if (!o) {
                Py_DECREF(out);
                return nullptr;
            }
            PyTuple_SET_ITEM(out, i, o);
        }
        return out;
    } catch (...) {
        return translate_exception();
    }
}

// current_stream(): the handle of torch's current stream
PyObject* py_current_stream(PyObject*, PyObject*) {
    try {
        return PyLong_FromVoidPtr(c10::cuda::getCurrentCUDAStream().stream());
    } catch (...) {
        return translate_exception();
    }
}

// bind(dispatch, combine, get_dispatch_layout, dispatch_sync): addresses of the library's entry points
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want_args(n, 4)) return nullptr;
    void* p[4];
    for (int i = 0; i < 4; ++i) {
        p[i] = PyLong_AsVoidPtr(a[i]);
        if (PyErr_Occurred()) return nullptr;
    }
    f_dispatch = reinterpret_cast<decltype(f_dispatch)>(p[0]);
    f_combine = reinterpret_cast<decltype(f_combine)>(p[1]);
    f_layout = reinterpret_cast<decltype(f_layout)>(p[2]);
    f_dispatch_sync = reinterpret_cast<decltype(f_dispatch_sync)>(p[3]);
    Py_RETURN_NONE;
}

#define UBEP_FAST(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(fn)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    UBEP_FAST("dispatch", py_dispatch),
    UBEP_FAST("dispatch_sync", py_dispatch_sync),
    UBEP_FAST("combine", py_combine),
    UBEP_FAST("combine_new", py_combine_new),
    UBEP_FAST("layout", py_layout),
    UBEP_FAST("layout_new", py_layout_new),
    UBEP_FAST("bind", py_bind),
    {"current_stream", py_current_stream, METH_NOARGS, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&kModule); }
