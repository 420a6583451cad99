// The per-token calls of binding.py as native functions: type and shape checks, output allocation, the current
// stream and the C-ABI call of include/spqt.h, without a Python-level step in between.  Argument marshalling
// only, like the ctypes path of the other calls.
//
// Why: a decode linear runs 4 to 10 us on the device, and marshalling it through Python and ctypes took 10 to
// 12 us per call (14 converted arguments, up to three torch.empty, one current_stream object, a checked
// data_ptr per tensor), so every small call was bound by the host.  In a stream of calls, before -> now: a
// 1024 x 4096 linear 13.7 -> 5.6 us, one index list and three 5120 x 5120 products 48.2 -> 22.9 us, the sixteen
// linears of four Llama-3-8B-shaped layers 175 -> 149 us (the device's own time in all three then; with later kernels 4.4, 15.8 and
// 115 us).
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/spqt.h"

namespace {

PyObject* g_error = nullptr;   // binding.SpqtError(status, where)

struct Names {
    PyObject *codes, *scale_zero, *records, *m, *n, *bits, *group, *cuda_stream;
} g_names;

// Leaves a call with a Python exception set.
struct Raised {};

[[noreturn]] void raise(PyObject* type, const char* fmt, const char* name)
{
    PyErr_Format(type, fmt, name);
    throw Raised();
}

void need_args(Py_ssize_t got, Py_ssize_t want)
{
    if (got != want) raise(PyExc_TypeError, "%s", "wrong number of arguments");
}

// The CUDA tensor behind a Python object, of the given type, contiguous; borrowed from `o`.
const at::Tensor& tensor_of(PyObject* o, at::ScalarType dtype, const char* name, bool contiguous = true)
{
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "%s must be a CUDA tensor", name);
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda()) raise(PyExc_TypeError, "%s must be a CUDA tensor", name);
    if (t.scalar_type() != dtype) {
        PyErr_Format(PyExc_TypeError, "%s must be %s, got %s", name, c10::toString(dtype), c10::toString(t.scalar_type()));
        throw Raised();
    }
    if (contiguous && !t.is_contiguous()) raise(PyExc_ValueError, "%s must be contiguous", name);
    return t;
}

// A tensor attribute of a packed matrix: the object keeps it alive for the call.
const at::Tensor& tensor_attr(PyObject* p, PyObject* attr, at::ScalarType dtype, const char* name)
{
    PyObject* o = PyObject_GetAttr(p, attr);
    if (!o) throw Raised();
    Py_DECREF(o);
    return tensor_of(o, dtype, name);
}

int int_attr(PyObject* p, PyObject* attr)
{
    PyObject* o = PyObject_GetAttr(p, attr);
    if (!o) throw Raised();
    const long v = PyLong_AsLong(o);
    Py_DECREF(o);
    if (v == -1 && PyErr_Occurred()) throw Raised();
    return (int)v;
}

int int_of(PyObject* o)
{
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised();
    return (int)v;
}

float float_of(PyObject* o)
{
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Raised();
    return (float)v;
}

void* stream_of(PyObject* o)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* s = PyObject_GetAttr(o, g_names.cuda_stream);
    if (!s) throw Raised();
    void* v = PyLong_AsVoidPtr(s);
    Py_DECREF(s);
    if (!v && PyErr_Occurred()) throw Raised();
    return v;
}

at::Tensor empty(at::IntArrayRef shape, at::ScalarType dtype, const at::Tensor& like)
{
    return at::detail::empty_cuda(shape, dtype, like.device(), std::nullopt);
}

// The tensor an optional argument names, or a new one.
at::Tensor given_or_empty(PyObject* o, at::IntArrayRef shape, at::ScalarType dtype, const char* name, const at::Tensor& like)
{
    return o == Py_None ? empty(shape, dtype, like) : tensor_of(o, dtype, name);
}

// A tensor argument as it goes back to the caller: the object that came in, or the new tensor.
PyObject* hand_back(PyObject* given, at::Tensor t)
{
    if (given != Py_None) {
        Py_INCREF(given);
        return given;
    }
    return THPVariable_Wrap(std::move(t));
}

// A tuple that takes over its items' references.
template <class... O>
PyObject* tuple_of(O... items)
{
    PyObject* const list[] = {items...};
    bool ok = true;
    for (PyObject* o : list) ok = ok && o;
    PyObject* t = ok ? PyTuple_New(sizeof...(items)) : nullptr;
    for (size_t i = 0; i < sizeof...(items); ++i) {
        if (t) PyTuple_SET_ITEM(t, (Py_ssize_t)i, list[i]);
        else Py_XDECREF(list[i]);
    }
    return t;
}

void check(spqt_status st, const char* where)
{
    if (st == SPQT_OK) return;
    PyObject* e = PyObject_CallFunction(g_error, "is", (int)st, where);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw Raised();
}

struct Zigzag {
    const void *codes, *scale_zero;
    int m, n, bits, group;
    explicit Zigzag(PyObject* p)
        : codes(tensor_attr(p, g_names.codes, at::kByte, "codes").data_ptr()),
          scale_zero(tensor_attr(p, g_names.scale_zero, at::kHalf, "scale_zero").data_ptr()),
          m(int_attr(p, g_names.m)), n(int_attr(p, g_names.n)), bits(int_attr(p, g_names.bits)), group(int_attr(p, g_names.group))
    {
    }
};

// Runs the library call without the GIL (a launch can wait for room in the stream's queue).
template <class F>
void call(const char* where, F f)
{
    spqt_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    check(st, where);
}

template <class F>
PyObject* guarded(F f)
{
    HANDLE_TH_ERRORS
    try {
        return f();
    } catch (const Raised&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

using Args = PyObject* const*;

// (x, t, idx, count, stream) -> (idx, count)
PyObject* sparsify(PyObject*, Args a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        need_args(na, 5);
        const at::Tensor& x = tensor_of(a[0], at::kHalf, "x");
        const float t = float_of(a[1]);
        const int64_t n = x.numel();
        at::Tensor idx = given_or_empty(a[2], {n > 0 ? n : 1}, at::kInt, "idx", x);
        at::Tensor count = given_or_empty(a[3], {1}, at::kInt, "count", x);
        if (idx.numel() < n) raise(PyExc_ValueError, "%s", "idx must hold n entries");
        void* s = stream_of(a[4]);
        call("spqt_sparsify", [&] { return spqt_sparsify(x.data_ptr(), (int)n, t, (int32_t*)idx.data_ptr(), (int32_t*)count.data_ptr(), s); });
        return tuple_of(hand_back(a[2], idx), hand_back(a[3], count));
    });
}

// (p, x, idx, count, workspace, y, stream) -> y
PyObject* sparse_gemv(PyObject*, Args a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        need_args(na, 7);
        const Zigzag p(a[0]);
        const at::Tensor& x = tensor_of(a[1], at::kHalf, "x");
        at::Tensor y = given_or_empty(a[5], {p.m}, at::kHalf, "y", x);
        if (x.numel() != p.n || y.numel() != p.m) raise(PyExc_ValueError, "%s", "x must have n entries and y m entries");
        const at::Tensor& idx = tensor_of(a[2], at::kInt, "idx");
        const at::Tensor& count = tensor_of(a[3], at::kInt, "count");
        const at::Tensor& ws = tensor_of(a[4], at::kByte, "workspace");
        void* s = stream_of(a[6]);
        call("spqt_sparse_gemv", [&] {
            return spqt_sparse_gemv(p.codes, p.scale_zero, p.m, p.n, p.bits, p.group, x.data_ptr(), (const int32_t*)idx.data_ptr(),
                                    (const int32_t*)count.data_ptr(), y.data_ptr(), ws.data_ptr(), (size_t)ws.numel(), s);
        });
        return hand_back(a[5], y);
    });
}

// (p, x, t, workspace, idx, count, y, stream) -> (y, idx, count)
PyObject* sparsify_gemv(PyObject*, Args a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        need_args(na, 8);
        const Zigzag p(a[0]);
        const at::Tensor& x = tensor_of(a[1], at::kHalf, "x");
        const float t = float_of(a[2]);
        const at::Tensor& ws = tensor_of(a[3], at::kByte, "workspace");
        at::Tensor idx = given_or_empty(a[4], {p.n}, at::kInt, "idx", x);
        at::Tensor count = given_or_empty(a[5], {1}, at::kInt, "count", x);
        at::Tensor y = given_or_empty(a[6], {p.m}, at::kHalf, "y", x);
        if (x.numel() != p.n || y.numel() != p.m || idx.numel() < p.n)
            raise(PyExc_ValueError, "%s", "x and idx must have n entries and y m entries");
        void* s = stream_of(a[7]);
        call("spqt_sparsify_gemv", [&] {
            return spqt_sparsify_gemv(p.codes, p.scale_zero, p.m, p.n, p.bits, p.group, x.data_ptr(), t, (int32_t*)idx.data_ptr(),
                                      (int32_t*)count.data_ptr(), y.data_ptr(), ws.data_ptr(), (size_t)ws.numel(), s);
        });
        return tuple_of(hand_back(a[6], y), hand_back(a[4], idx), hand_back(a[5], count));
    });
}

// (p, x, workspace, y, stream) -> y
PyObject* dense_gemv(PyObject*, Args a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        need_args(na, 5);
        const Zigzag p(a[0]);
        const at::Tensor& x = tensor_of(a[1], at::kHalf, "x");
        at::Tensor y = given_or_empty(a[3], {p.m}, at::kHalf, "y", x);
        if (x.numel() != p.n || y.numel() != p.m) raise(PyExc_ValueError, "%s", "x must have n entries and y m entries");
        const at::Tensor& ws = tensor_of(a[2], at::kByte, "workspace");
        void* s = stream_of(a[4]);
        call("spqt_dense_gemv", [&] {
            return spqt_dense_gemv(p.codes, p.scale_zero, p.m, p.n, p.bits, p.group, x.data_ptr(), y.data_ptr(), ws.data_ptr(),
                                   (size_t)ws.numel(), s);
        });
        return hand_back(a[3], y);
    });
}

// X [batch <= 8][n] with unit column stride, and Y [batch][m], given or new
at::Tensor batch_output(const Zigzag& p, PyObject* X_o, PyObject* Y_o)
{
    if (!THPVariable_Check(X_o)) raise(PyExc_TypeError, "%s", "X and Y must be CUDA float16 tensors");
    const at::Tensor& X = THPVariable_Unpack(X_o);
    if (X.dim() != 2 || X.stride(1) != 1 || X.size(1) != p.n || X.size(0) < 1 || X.size(0) > 8)
        raise(PyExc_ValueError, "%s", "X must be [batch <= 8][n] with unit column stride");
    if (X.scalar_type() != at::kHalf || !X.is_cuda()) raise(PyExc_TypeError, "%s", "X and Y must be CUDA float16 tensors");
    if (Y_o == Py_None) return empty({X.size(0), p.m}, at::kHalf, X);
    if (!THPVariable_Check(Y_o)) raise(PyExc_TypeError, "%s", "X and Y must be CUDA float16 tensors");
    const at::Tensor& Y = THPVariable_Unpack(Y_o);
    if (Y.scalar_type() != at::kHalf || !Y.is_cuda()) raise(PyExc_TypeError, "%s", "X and Y must be CUDA float16 tensors");
    if (Y.dim() != 2 || Y.size(0) != X.size(0) || Y.size(1) != p.m || Y.stride(1) != 1)
        raise(PyExc_ValueError, "%s", "Y must be [batch][m] with unit column stride");
    return Y;
}

// (p, X, t, workspace, idx, count, Y, stream) -> (Y, idx, count)
PyObject* sparse_gemm_small(PyObject*, Args a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        need_args(na, 8);
        const Zigzag p(a[0]);
        at::Tensor Y = batch_output(p, a[1], a[6]);
        const at::Tensor& X = THPVariable_Unpack(a[1]);
        const float t = float_of(a[2]);
        const at::Tensor& ws = tensor_of(a[3], at::kByte, "workspace");
        at::Tensor idx = given_or_empty(a[4], {p.n}, at::kInt, "idx", X);
        at::Tensor count = given_or_empty(a[5], {1}, at::kInt, "count", X);
        void* s = stream_of(a[7]);
        call("spqt_sparse_gemm_small", [&] {
            return spqt_sparse_gemm_small(p.codes, p.scale_zero, p.m, p.n, p.bits, p.group, X.data_ptr(), (int)X.stride(0), (int)X.size(0), t,
                                          (int32_t*)idx.data_ptr(), (int32_t*)count.data_ptr(), Y.data_ptr(), (int)Y.stride(0), ws.data_ptr(),
                                          (size_t)ws.numel(), s);
        });
        return tuple_of(hand_back(a[6], Y), hand_back(a[4], idx), hand_back(a[5], count));
    });
}

// (p, X, workspace, Y, stream) -> Y
PyObject* dense_gemm_small(PyObject*, Args a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        need_args(na, 5);
        const Zigzag p(a[0]);
        at::Tensor Y = batch_output(p, a[1], a[3]);
        const at::Tensor& X = THPVariable_Unpack(a[1]);
        const at::Tensor& ws = tensor_of(a[2], at::kByte, "workspace");
        void* s = stream_of(a[4]);
        call("spqt_dense_gemm_small", [&] {
            return spqt_dense_gemm_small(p.codes, p.scale_zero, p.m, p.n, p.bits, p.group, X.data_ptr(), (int)X.stride(0), (int)X.size(0),
                                         Y.data_ptr(), (int)Y.stride(0), ws.data_ptr(), (size_t)ws.numel(), s);
        });
        return hand_back(a[3], Y);
    });
}

// list: (p, x, idx, count, workspace, y, stream, where) -> y; over all columns: without idx and count
template <bool LIST>
PyObject* kqw_gemv(PyObject*, Args a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        need_args(na, LIST ? 8 : 6);
        PyObject* p = a[0];
        const Args rest = a + (LIST ? 4 : 2);   // workspace, y, stream, where
        const void* records = tensor_attr(p, g_names.records, at::kByte, "records").data_ptr();
        const int m = int_attr(p, g_names.m), n = int_attr(p, g_names.n), bits = int_attr(p, g_names.bits);
        const at::Tensor& x = tensor_of(a[1], at::kHalf, "x");
        at::Tensor y = given_or_empty(rest[1], {m}, at::kHalf, "y", x);
        const at::Tensor& ws = tensor_of(rest[0], at::kByte, "workspace");
        void* s = stream_of(rest[2]);
        const char* where = PyUnicode_AsUTF8(rest[3]);
        if (!where) throw Raised();
        if (LIST) {
            const at::Tensor& idx = tensor_of(a[2], at::kInt, "idx");
            const at::Tensor& count = tensor_of(a[3], at::kInt, "count");
            call(where, [&] {
                return spqt_kqw_sparse_gemv(records, m, n, bits, x.data_ptr(), (const int32_t*)idx.data_ptr(), (const int32_t*)count.data_ptr(),
                                            y.data_ptr(), ws.data_ptr(), (size_t)ws.numel(), s);
            });
        } else {
            call(where, [&] { return spqt_kqw_dense_gemv(records, m, n, bits, x.data_ptr(), y.data_ptr(), ws.data_ptr(), (size_t)ws.numel(), s); });
        }
        return hand_back(rest[1], y);
    });
}

constexpr auto kqw_sparse_gemv = kqw_gemv<true>;
constexpr auto kqw_dense_gemv = kqw_gemv<false>;

const at::Tensor& weights_of(PyObject* o)
{
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "%s", "W must be a CUDA float16 tensor");
    const at::Tensor& W = THPVariable_Unpack(o);
    if (W.dim() != 2 || W.stride(1) != 1) raise(PyExc_ValueError, "%s", "W must be 2-D with unit column stride");
    if (!W.is_cuda() || W.scalar_type() != at::kHalf) raise(PyExc_TypeError, "%s", "W must be a CUDA float16 tensor");
    return W;
}

// (W, bits, group, stream) -> (codes, scale_zero)
PyObject* pack(PyObject*, Args a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        need_args(na, 4);
        const at::Tensor& W = weights_of(a[0]);
        const int m = (int)W.size(0), n = (int)W.size(1), bits = int_of(a[1]), group = int_of(a[2]);
        size_t cb = 0, sb = 0;
        check(spqt_packed_sizes(m, n, bits, group, &cb, &sb, nullptr), "spqt_packed_sizes");
        at::Tensor codes = empty({(int64_t)cb}, at::kByte, W), sz = empty({(int64_t)(sb / 2)}, at::kHalf, W);
        void* s = stream_of(a[3]);
        call("spqt_pack", [&] { return spqt_pack(W.data_ptr(), m, n, (int)W.stride(0), bits, group, codes.data_ptr(), sz.data_ptr(), s); });
        return tuple_of(hand_back(Py_None, codes), hand_back(Py_None, sz));
    });
}

// (W, bits, stream, where) -> records
PyObject* kqw_pack(PyObject*, Args a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        need_args(na, 4);
        const at::Tensor& W = weights_of(a[0]);
        const int m = (int)W.size(0), n = (int)W.size(1), bits = int_of(a[1]);
        const char* where = PyUnicode_AsUTF8(a[3]);
        if (!where) throw Raised();
        size_t rb = 0;
        check(spqt_kqw_packed_sizes(m, n, bits, &rb, nullptr), "spqt_kqw_packed_sizes");
        at::Tensor records = empty({(int64_t)rb}, at::kByte, W);
        void* s = stream_of(a[2]);
        call(where, [&] { return spqt_kqw_pack(W.data_ptr(), m, n, (int)W.stride(0), bits, records.data_ptr(), s); });
        return hand_back(Py_None, records);
    });
}

// (handle, stream)
PyObject* host_step_launch(PyObject*, Args a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        need_args(na, 2);
        void* step = a[0] == Py_None ? nullptr : PyLong_AsVoidPtr(a[0]);
        if (!step && PyErr_Occurred()) throw Raised();
        void* s = stream_of(a[1]);
        call("spqt_host_step_launch", [&] { return spqt_host_step_launch(step, s); });
        Py_RETURN_NONE;
    });
}

PyObject* set_error(PyObject*, PyObject* cls)
{
    Py_INCREF(cls);
    Py_XSETREF(g_error, cls);
    Py_RETURN_NONE;
}

#define SPQT_METHOD(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    SPQT_METHOD(sparsify), SPQT_METHOD(sparse_gemv), SPQT_METHOD(sparsify_gemv), SPQT_METHOD(dense_gemv),
    SPQT_METHOD(sparse_gemm_small), SPQT_METHOD(dense_gemm_small), SPQT_METHOD(kqw_sparse_gemv), SPQT_METHOD(kqw_dense_gemv), SPQT_METHOD(pack),
    SPQT_METHOD(kqw_pack), SPQT_METHOD(host_step_launch),
    {"set_error", set_error, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void)
{
    g_names = {PyUnicode_InternFromString("codes"), PyUnicode_InternFromString("scale_zero"), PyUnicode_InternFromString("records"),
               PyUnicode_InternFromString("m"), PyUnicode_InternFromString("n"), PyUnicode_InternFromString("bits"),
               PyUnicode_InternFromString("group"), PyUnicode_InternFromString("cuda_stream")};
    return PyModule_Create(&g_module);
}
