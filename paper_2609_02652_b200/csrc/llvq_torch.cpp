// The calls of binding.py that a serving loop makes, in native code: torch tensors -> the C entry points of llvq.h.
// Argument checks, the current stream and the output's allocation cost a few hundred nanoseconds here; through Python
// and ctypes they took 9 us of a 13 us call, more than the matvec itself up to 8192 x 8192.
//
// Nothing is computed.  The entry points' addresses come from the library that binding.py has loaded (bind()).
#include <Python.h>

#include <ATen/Context.h>
#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <ATen/ops/empty.h>
#include <ATen/record_function.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/llvq.h"

namespace {

#define LLVQ_TORCH_CALLS(X)                                                                                              \
    X(llvq_gemv) X(llvq_gemv_batch) X(llvq_gemv_grouped) X(llvq_gemv_rotated) X(llvq_gemv_static) X(llvq_gemv_fp16)      \
    X(llvq_gemv_noweights) X(llvq_rotate) X(llvq_expand) X(llvq_overlay_count) X(llvq_dequant_fp16) X(llvq_layout_bytes)
#define LLVQ_TORCH_POINTER(name) decltype(&::name) name = nullptr;
struct Entry {
    LLVQ_TORCH_CALLS(LLVQ_TORCH_POINTER)
} entry;
PyObject *error_class = nullptr;
PyObject *handle_name = nullptr, *cuda_stream_name = nullptr;
PyObject *gain_index[2] = {nullptr, nullptr};

// ---- arguments
int64_t integer(PyObject *o) {
    if (!PyLong_Check(o)) {                        // as int(o)
        PyObject *n = PyNumber_Long(o);
        if (!n) throw python_error();
        const int64_t v = PyLong_AsLongLong(n);
        Py_DECREF(n);
        if (v == -1 && PyErr_Occurred()) throw python_error();
        return v;
    }
    const int64_t v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw python_error();
    return v;
}

llvq_ctx *context(PyObject *o) {
    PyObject *h = PyObject_GetAttr(o, handle_name);
    if (!h) throw python_error();
    void *p = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!p) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, "context already destroyed");
        throw python_error();
    }
    return static_cast<llvq_ctx *>(p);
}

const char *dtype_name(at::ScalarType t) {
    switch (t) {
        case at::kHalf: return "torch.float16";
        case at::kFloat: return "torch.float32";
        case at::kLong: return "torch.int64";
        case at::kInt: return "torch.int32";
        default: return "torch.uint8";
    }
}
const at::Tensor &tensor(PyObject *o, at::ScalarType dtype, const char *what) {
    if (THPVariable_Check(o)) {
        const at::Tensor &t = THPVariable_Unpack(o);
        if (t.is_cuda() && t.scalar_type() == dtype && t.is_contiguous()) return t;
    }
    PyErr_Format(PyExc_TypeError, "%s: expected a contiguous CUDA tensor of dtype %s", what, dtype_name(dtype));
    throw python_error();
}
template <typename T = void>
T *device_pointer(PyObject *o, at::ScalarType dtype, const char *what) { return static_cast<T *>(tensor(o, dtype, what).data_ptr()); }

// float(o[0]), float(o[1]), whatever o indexes by 0 and 1: a tuple, an array, a tensor (which is no sequence to Python's C API)
struct Gain {
    float v[2];
    explicit Gain(PyObject *o) {
        for (int i = 0; i < 2; i++) {
            PyObject *item = PyObject_GetItem(o, gain_index[i]);
            if (!item) throw python_error();
            PyObject *number = PyFloat_CheckExact(item) ? item : PyNumber_Float(item);
            if (number != item) Py_DECREF(item);
            if (!number) throw python_error();
            v[i] = static_cast<float>(PyFloat_AS_DOUBLE(number));
            Py_DECREF(number);
        }
    }
};

void *stream(PyObject *o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject *s = PyObject_GetAttr(o, cuda_stream_name);
    if (!s) throw python_error();
    void *p = PyLong_AsVoidPtr(s);
    Py_DECREF(s);
    if (!p && PyErr_Occurred()) throw python_error();
    return p;
}

// torch.empty.  Where nothing in this thread could act on the call - no dispatch mode, transform, inference mode or profiler,
// no fill under deterministic algorithms - the allocation alone is made: the dispatcher takes 0.35 us of a call of 4.4 (1024 x 2560,
// back to back), its CUDA kernel alone still 0.25.
at::Tensor new_tensor(at::IntArrayRef shape, at::ScalarType dtype, c10::Device device) {
    const bool plain = c10::impl::tls_local_dispatch_key_set().included_ == c10::default_included_set && !at::hasCallbacks() &&
                       !at::globalContext().deterministicAlgorithms();
    return plain ? at::Tensor(at::detail::empty_cuda(shape, dtype, device, std::nullopt)) : at::empty(shape, at::TensorOptions().dtype(dtype).device(device));
}

// An output: the tensor the caller gave (checked), or a new one on the device of `like`.
struct Output {
    PyObject *object;        // owned
    void *data;
    Output(PyObject *given, at::IntArrayRef shape, at::ScalarType dtype, const at::Tensor &like, const char *what) {
        if (given != Py_None) {
            data = device_pointer(given, dtype, what);
            Py_INCREF(given);
            object = given;
        } else {
            at::Tensor t = new_tensor(shape, dtype, like.device());
            data = t.data_ptr();
            object = THPVariable_Wrap(std::move(t));
            if (!object) throw python_error();
        }
    }
    ~Output() { Py_XDECREF(object); }
    PyObject *release() { PyObject *o = object; object = nullptr; return o; }
};

// Calls a C entry point without the interpreter lock (a launch blocks while the stream's queue is full) and turns an
// error code into the binding's exception.
template <typename F>
void call(const char *what, F f) {
    int code;
    Py_BEGIN_ALLOW_THREADS
    code = f();
    Py_END_ALLOW_THREADS
    if (code != LLVQ_OK) {
        PyObject *e = PyObject_CallFunction(error_class, "is", code, what);
        if (e) {
            PyErr_SetObject(error_class, e);
            Py_DECREF(e);
        }
        throw python_error();
    }
}

// A host array of llvq_problem (the ctypes array of make_problems).
struct Problems {
    Py_buffer view;
    explicit Problems(PyObject *o) {
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw python_error();
    }
    ~Problems() { PyBuffer_Release(&view); }
    const llvq_problem *data() const { return static_cast<const llvq_problem *>(view.buf); }
    int count() const { return static_cast<int>(view.len / (Py_ssize_t)sizeof(llvq_problem)); }
};

// ---- the calls; arguments in the order of binding.py, None where it has a default of None
PyObject *gemv(PyObject *const *a) {
    llvq_ctx *ctx = context(a[0]);
    const int layout = (int)integer(a[1]);
    const void *buf = device_pointer(a[2], at::kByte, "layout_buf"), *scale = device_pointer(a[3], at::kHalf, "row_scale");
    const Gain gain(a[4]);
    const at::Tensor &x = tensor(a[5], at::kHalf, "x");
    const int64_t rows = integer(a[6]), k = integer(a[7]);
    Output y(a[8], {rows}, at::kFloat, x, "y");
    void *s = stream(a[9]);
    call("llvq_gemv", [&] { return entry.llvq_gemv(ctx, layout, buf, scale, gain.v, x.data_ptr(), (float *)y.data, rows, k, s); });
    return y.release();
}

PyObject *gemv_batch(PyObject *const *a) {
    llvq_ctx *ctx = context(a[0]);
    const void *buf = device_pointer(a[1], at::kByte, "layout_buf"), *scale = device_pointer(a[2], at::kHalf, "row_scale");
    const Gain gain(a[3]);
    const int64_t rows = integer(a[5]), k = integer(a[6]);
    if (!THPVariable_Check(a[4]) || THPVariable_Unpack(a[4]).dim() != 2 || THPVariable_Unpack(a[4]).size(1) != k ||
        !THPVariable_Unpack(a[4]).is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "x must be a contiguous [batch, k_padded] tensor");
        throw python_error();
    }
    const at::Tensor &x = tensor(a[4], at::kHalf, "x");
    const int64_t batch = x.size(0);
    Output y(a[7], {batch, rows}, at::kFloat, x, "y");
    void *s = stream(a[8]);
    call("llvq_gemv_batch", [&] { return entry.llvq_gemv_batch(ctx, buf, scale, gain.v, x.data_ptr(), (float *)y.data, rows, k, (int)batch, s); });
    return y.release();
}

PyObject *gemv_static(PyObject *const *a) {
    const void *buf = device_pointer(a[0], at::kByte, "layout_buf"), *scale = device_pointer(a[1], at::kHalf, "row_scale");
    const Gain gain(a[2]);
    const void *x = device_pointer(a[3], at::kHalf, "x");
    const int64_t rows = integer(a[4]), k = integer(a[5]);
    float *y = device_pointer<float>(a[6], at::kFloat, "y");
    void *s = stream(a[7]);
    call("llvq_gemv_static", [&] { return entry.llvq_gemv_static(buf, scale, gain.v, x, y, rows, k, s); });
    Py_INCREF(a[6]);
    return a[6];
}

PyObject *gemv_grouped(PyObject *const *a) {
    llvq_ctx *ctx = context(a[0]);
    const int layout = (int)integer(a[1]);
    const Problems problems(a[2]);
    const void *x = device_pointer(a[3], at::kHalf, "x");
    const int64_t k = integer(a[4]);
    void *s = stream(a[5]);
    call("llvq_gemv_grouped", [&] { return entry.llvq_gemv_grouped(ctx, layout, problems.data(), problems.count(), x, k, s); });
    Py_RETURN_NONE;
}

PyObject *gemv_rotated(PyObject *const *a) {
    llvq_ctx *ctx = context(a[0]);
    const Problems problems(a[1]);
    const void *x = device_pointer(a[2], at::kHalf, "x");
    const int64_t k = integer(a[3]);
    llvq_rotation rot;
    rot.n = integer(a[4]);
    rot.block = integer(a[5]);
    rot.negate_bits = a[6] == Py_None ? nullptr : device_pointer<const uint32_t>(a[6], at::kInt, "negate_bits");
    void *s = stream(a[7]);
    call("llvq_gemv_rotated", [&] { return entry.llvq_gemv_rotated(ctx, problems.data(), problems.count(), x, k, &rot, s); });
    Py_RETURN_NONE;
}

PyObject *gemv_fp16(PyObject *const *a) {
    const void *W = device_pointer(a[0], at::kHalf, "W");
    const at::Tensor &x = tensor(a[1], at::kHalf, "x");
    const int64_t rows = integer(a[2]), k = integer(a[3]);
    Output y(a[4], {rows}, at::kFloat, x, "y");
    void *s = stream(a[5]);
    call("llvq_gemv_fp16", [&] { return entry.llvq_gemv_fp16(W, x.data_ptr(), (float *)y.data, rows, k, s); });
    return y.release();
}

PyObject *gemv_noweights(PyObject *const *a) {
    llvq_ctx *ctx = context(a[0]);
    const void *scale = device_pointer(a[1], at::kHalf, "row_scale");
    const at::Tensor &x = tensor(a[2], at::kHalf, "x");
    const int64_t rows = integer(a[3]), k = integer(a[4]);
    Output y(a[5], {rows}, at::kFloat, x, "y");
    void *s = stream(a[6]);
    call("llvq_gemv_noweights", [&] { return entry.llvq_gemv_noweights(ctx, scale, x.data_ptr(), (float *)y.data, rows, k, s); });
    return y.release();
}

PyObject *rotate(PyObject *const *a) {
    llvq_ctx *ctx = context(a[0]);
    const at::Tensor &x = tensor(a[1], at::kHalf, "x");
    const int64_t block = integer(a[2]);
    const uint32_t *negate = a[3] == Py_None ? nullptr : device_pointer<const uint32_t>(a[3], at::kInt, "negate_bits");
    Output y(a[4], x.sizes(), at::kHalf, x, "y");
    void *s = stream(a[5]);
    call("llvq_rotate", [&] { return entry.llvq_rotate(ctx, x.data_ptr(), y.data, negate, x.numel(), block, s); });
    return y.release();
}

PyObject *expand(PyObject *const *a) {
    llvq_ctx *ctx = context(a[0]);
    const int layout = (int)integer(a[1]);
    const at::Tensor &codes = tensor(a[2], at::kLong, "codes");
    const int64_t rows = integer(a[3]), nb = integer(a[4]);
    size_t bytes = 0;
    if (a[5] == Py_None) call("llvq_layout_bytes", [&] { return entry.llvq_layout_bytes(layout, rows, nb * 24, &bytes); });
    Output out(a[5], {(int64_t)bytes}, at::kByte, codes, "out");
    if (a[5] != Py_None) bytes = (size_t)THPVariable_Unpack(a[5]).numel();
    uint32_t *bad = a[6] == Py_None ? nullptr : device_pointer<uint32_t>(a[6], at::kInt, "bad_count");
    void *s = stream(a[7]);
    call("llvq_expand", [&] { return entry.llvq_expand(ctx, layout, (const uint64_t *)codes.data_ptr(), rows, nb, out.data, bytes, bad, s); });
    return out.release();
}

PyObject *overlay_count(PyObject *const *a) {
    llvq_ctx *ctx = context(a[0]);
    const uint64_t *codes = device_pointer<const uint64_t>(a[1], at::kLong, "codes");
    const int64_t rows = integer(a[2]), nb = integer(a[3]);
    void *s = stream(a[4]);
    uint64_t count = 0;
    call("llvq_overlay_count", [&] { return entry.llvq_overlay_count(ctx, codes, rows, nb, &count, s); });
    return PyLong_FromUnsignedLongLong(count);
}

PyObject *dequant_fp16(PyObject *const *a) {
    llvq_ctx *ctx = context(a[0]);
    const int layout = (int)integer(a[1]);
    const at::Tensor &buf = tensor(a[2], at::kByte, "layout_buf");
    const void *scale = device_pointer(a[3], at::kHalf, "row_scale");
    const Gain gain(a[4]);
    const int64_t rows = integer(a[5]), k = integer(a[6]);
    Output W(a[7], {rows, k}, at::kHalf, buf, "W");
    void *s = stream(a[8]);
    call("llvq_dequant_fp16", [&] { return entry.llvq_dequant_fp16(ctx, layout, buf.data_ptr(), scale, gain.v, W.data, rows, k, s); });
    return W.release();
}

// ---- Python's side
template <PyObject *(*F)(PyObject *const *), int N>
PyObject *method(PyObject *, PyObject *const *args, Py_ssize_t n) {
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "%d arguments expected, %zd given", N, n);
        return nullptr;
    }
    HANDLE_TH_ERRORS
    return F(args);
    END_HANDLE_TH_ERRORS
}

// bind(exception class, {entry point's name: address})
PyObject *bind(PyObject *, PyObject *args) {
    PyObject *cls, *addresses;
    if (!PyArg_ParseTuple(args, "OO!", &cls, &PyDict_Type, &addresses)) return nullptr;
    Entry e;
#define LLVQ_TORCH_BIND(name)                                                                    \
    {                                                                                            \
        PyObject *p = PyDict_GetItemString(addresses, #name);                                    \
        e.name = p ? reinterpret_cast<decltype(&::name)>(PyLong_AsVoidPtr(p)) : nullptr;         \
        if (!e.name) return PyErr_Format(PyExc_RuntimeError, "no address for %s", #name);        \
    }
    LLVQ_TORCH_CALLS(LLVQ_TORCH_BIND)
    entry = e;
    Py_INCREF(cls);
    Py_XSETREF(error_class, cls);
    Py_RETURN_NONE;
}

template <PyObject *(*F)(PyObject *const *), int N>
PyMethodDef fast(const char *name) { return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&method<F, N>)), METH_FASTCALL, nullptr}; }

PyMethodDef methods[] = {fast<gemv, 10>("gemv"), fast<gemv_batch, 9>("gemv_batch"), fast<gemv_static, 8>("gemv_static"),
                         fast<gemv_grouped, 6>("gemv_grouped"), fast<gemv_rotated, 8>("gemv_rotated"), fast<gemv_fp16, 6>("gemv_fp16"),
                         fast<gemv_noweights, 7>("gemv_noweights"), fast<rotate, 6>("rotate"), fast<expand, 8>("expand"),
                         fast<overlay_count, 5>("overlay_count"), fast<dequant_fp16, 9>("dequant_fp16"),
                         {"bind", bind, METH_VARARGS, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() {
    handle_name = PyUnicode_InternFromString("handle");
    cuda_stream_name = PyUnicode_InternFromString("cuda_stream");
    for (int i = 0; i < 2; i++) gain_index[i] = PyLong_FromLong(i);
    if (!handle_name || !cuda_stream_name || !gain_index[0] || !gain_index[1]) return nullptr;
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", LLVQ_BUILT_FOR) != 0) Py_CLEAR(m);
    return m;
}
