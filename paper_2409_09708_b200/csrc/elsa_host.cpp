// The calls of binding.py whose launch takes the device no longer than Python takes to make it, as one native call each:
// arguments unpacked, outputs allocated by torch's allocator, the library's entry point called.  No arithmetic.
//
// A layer of one image (197 x 768 -> 768) is 3.5 us of device time.  Through ctypes a call took 8.6 us of host time: 2.5 in
// the library, 1.3 in the conversion of 15 arguments, 1.8 for the output tensor, the rest Python; four levels of a
// 3072 x 768 weight took 20.7, half of it views of the two allocations.
//
// Every function returns its result, or the entry point's status as an int when that is not ELSA_OK (binding.py raises).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/EmptyTensor.h>
#include <c10/core/impl/DeviceGuardImplInterface.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <torch/csrc/autograd/python_variable.h>

#include "elsa.h"

namespace {

decltype(&elsa_nm_linear) g_linear;
decltype(&elsa_nm_linear_masked) g_linear_masked;
decltype(&elsa_nm_linear_i8) g_linear_i8;
decltype(&elsa_nm_linear_backward) g_backward;
decltype(&elsa_nm_compress) g_compress;
decltype(&elsa_nm_compress_levels) g_compress_levels;
decltype(&elsa_nm_values_bytes) g_values_bytes;
decltype(&elsa_nm_index_bytes) g_index_bytes;
decltype(&elsa_workspace_bytes) g_workspace_bytes;
decltype(&elsa_workspace_bytes_i8) g_workspace_bytes_i8;
decltype(&elsa_backward_workspace_bytes) g_backward_workspace_bytes;

// What a conversion found wrong; the Python error is set.
struct Raised {};

const at::Tensor& tensor(PyObject* o)
{
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "tensor expected, got %s", Py_TYPE(o)->tp_name);
        throw Raised();
    }
    return THPVariable_Unpack(o);
}

void* pointer(const at::Tensor& t)
{
    if (!t.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "contiguous tensor expected");
        throw Raised();
    }
    return t.data_ptr();
}

void* pointer(PyObject* o) { return o == Py_None ? nullptr : pointer(tensor(o)); }

int integer(PyObject* o)
{
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised();
    return (int)v;
}

void* handle(PyObject* o)
{
    if (o == Py_None) return nullptr;
    void* p = PyLong_AsVoidPtr(o);
    if (p == nullptr && PyErr_Occurred()) throw Raised();
    return p;
}

int64_t size_at(const at::Tensor& t, int64_t dim)
{
    if (dim >= t.dim()) {
        PyErr_SetString(PyExc_IndexError, "tensor has too few dimensions");
        throw Raised();
    }
    return t.size(dim);
}

// A tensor read as a matrix: a third dimension would be dropped without a word.
const at::Tensor& matrix(PyObject* o)
{
    const at::Tensor& t = tensor(o);
    if (t.dim() != 2) {
        PyErr_Format(t.dim() < 2 ? PyExc_IndexError : PyExc_ValueError, "tensor of two dimensions expected, got %d", (int)t.dim());
        throw Raised();
    }
    return t;
}

// A new tensor of this shape beside `like`.  On the current GPU straight from torch's current CUDA allocator (the one that
// torch.cuda.memory.change_current_allocator puts in place; c10::GetAllocator keeps the built-in one): by way of at::empty's dispatch
// eight outputs, four levels of a weight, were most of the call (3072 x 768 11.5 us with it, 9.4 without).  What at::empty
// does besides is left to it: another device, filled memory, and whatever takes part in a call on this thread beyond the ordinary
// (dispatch modes, functional transforms, tracing), which shows as a dispatch key included.
at::Tensor fresh(const at::Tensor& like, at::IntArrayRef shape, at::ScalarType type)
{
    const c10::Device device = like.device();
    const at::Context& context = at::globalContext();
    if (device.is_cuda() && c10::impl::getDeviceGuardImpl(c10::DeviceType::CUDA)->getDevice() == device &&
        (c10::impl::tls_local_dispatch_key_set().included_ - c10::default_included_set).empty() && !(context.deterministicAlgorithms() && context.deterministicFillUninitializedMemory()))
        return at::detail::empty_generic(shape, c10::cuda::CUDACachingAllocator::get(), c10::DispatchKeySet(c10::DispatchKey::CUDA), type, std::nullopt);
    return at::empty(shape, like.options().dtype(type));
}

// The given tensor, or a new one of this shape beside `like`.
at::Tensor given_or_new(PyObject* o, const at::Tensor& like, at::IntArrayRef shape, at::ScalarType type)
{
    return o != Py_None ? tensor(o) : fresh(like, shape, type);
}

// A workspace of at least `bytes`.
at::Tensor workspace(PyObject* o, const at::Tensor& like, size_t bytes)
{
    return given_or_new(o, like, {(int64_t)(bytes < 256 ? 256 : bytes)}, at::kByte);
}

PyObject* result_or_status(elsa_status st, const at::Tensor& t)
{
    return st == ELSA_OK ? THPVariable_Wrap(t) : PyLong_FromLong((long)st);
}

// C++ exceptions (torch's among them) become Python errors; n: the arguments expected.
template <typename F>
PyObject* guarded(Py_ssize_t got, Py_ssize_t n, F f)
{
    if (got != n) return PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", n, got);
    try {
        return f();
    } catch (const Raised&) {
        return nullptr;
    } catch (const c10::Error& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// The entry point without the interpreter's lock.
template <typename F>
elsa_status unlocked(F f)
{
    elsa_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return st;
}

// X, vals, idx, bias, out, in, N, M, dtype code, Y, workspace, dev_status, stream
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded(n, 13, [&] {
        const at::Tensor& X = tensor(a[0]);
        const int rows = (int)size_at(X, 0), out = integer(a[4]), in = integer(a[5]), N = integer(a[6]), M = integer(a[7]);
        const elsa_dtype code = (elsa_dtype)integer(a[8]);
        const at::Tensor Y = given_or_new(a[9], X, {rows, out}, X.scalar_type());
        const at::Tensor ws = workspace(a[10], X, a[10] == Py_None ? g_workspace_bytes(rows, in, out, N, M, code) : 0);
        void *x = pointer(X), *vals = pointer(a[1]), *idx = pointer(a[2]), *bias = pointer(a[3]), *y = pointer(Y), *w = pointer(ws),
             *status = pointer(a[11]), *stream = handle(a[12]);
        const size_t bytes = (size_t)ws.numel();
        return result_or_status(unlocked([&] {
            return g_linear(x, rows, vals, (const uint32_t*)idx, bias, out, in, N, M, code, y, w, bytes, (uint32_t*)status, stream);
        }), Y);
    });
}

// X, W, bias, N, M, dtype code, Y, workspace, dev_status, stream
PyObject* linear_masked(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded(n, 10, [&] {
        const at::Tensor &X = matrix(a[0]), &W = matrix(a[1]);
        const int rows = (int)size_at(X, 0), in = (int)size_at(X, 1), out = (int)size_at(W, 0), N = integer(a[3]), M = integer(a[4]);
        const elsa_dtype code = (elsa_dtype)integer(a[5]);
        const at::Tensor Y = given_or_new(a[6], X, {rows, out}, X.scalar_type());
        const at::Tensor ws = workspace(a[7], X, a[7] == Py_None ? g_workspace_bytes(rows, in, out, N, M, code) : 0);
        void *x = pointer(X), *wm = pointer(W), *bias = pointer(a[2]), *y = pointer(Y), *w = pointer(ws), *status = pointer(a[8]),
             *stream = handle(a[9]);
        const size_t bytes = (size_t)ws.numel();
        return result_or_status(unlocked([&] {
            return g_linear_masked(x, rows, wm, bias, out, in, N, M, code, y, w, bytes, (uint32_t*)status, stream);
        }), Y);
    });
}

// X, x_scale, vals, idx, w_scale, bias, out, in, N, M, dtype code of Y, dev_status, stream
PyObject* linear_i8(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded(n, 13, [&] {
        const at::Tensor& X = tensor(a[0]);
        const double x_scale = PyFloat_AsDouble(a[1]);
        if (x_scale == -1.0 && PyErr_Occurred()) throw Raised();
        const int rows = (int)size_at(X, 0), out = integer(a[6]), in = integer(a[7]), N = integer(a[8]), M = integer(a[9]), code = integer(a[10]);
        const at::Tensor Y = fresh(X, {rows, out}, code == ELSA_BF16 ? at::kBFloat16 : at::kHalf);
        const size_t need = g_workspace_bytes_i8(out, in, N, M);
        at::Tensor ws;
        if (need > 0) ws = workspace(Py_None, X, need);
        void *x = pointer(X), *vals = pointer(a[2]), *idx = pointer(a[3]), *scale = pointer(a[4]), *bias = pointer(a[5]), *y = pointer(Y),
             *w = need > 0 ? ws.data_ptr() : nullptr, *status = pointer(a[11]), *stream = handle(a[12]);
        return result_or_status(unlocked([&] {
            return g_linear_i8((const int8_t*)x, rows, (float)x_scale, (const int8_t*)vals, (const uint32_t*)idx, (const float*)scale, bias, out,
                               in, N, M, (elsa_dtype)code, y, w, need, (uint32_t*)status, stream);
        }), Y);
    });
}

// dY, X, vals, idx, out, in, N, M, dtype code, dX wanted, dW wanted, db wanted, workspace, dev_status, stream -> (dX, dW, db)
PyObject* linear_backward(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded(n, 15, [&]() -> PyObject* {
        const at::Tensor& dY = tensor(a[0]);
        const int rows = (int)size_at(dY, 0), out = integer(a[4]), in = integer(a[5]), N = integer(a[6]), M = integer(a[7]);
        const elsa_dtype code = (elsa_dtype)integer(a[8]);
        at::Tensor grad[3];
        const int64_t shape[3][2] = {{rows, in}, {out, in}, {out, 1}};
        void* g[3] = {nullptr, nullptr, nullptr};
        for (int i = 0; i < 3; ++i) {
            const int wanted = PyObject_IsTrue(a[9 + i]);
            if (wanted < 0) throw Raised();
            if (!wanted) continue;
            grad[i] = fresh(dY, at::IntArrayRef(shape[i], i == 2 ? 1 : 2), dY.scalar_type());
            g[i] = grad[i].data_ptr();
        }
        const at::Tensor ws = workspace(a[12], dY, a[12] == Py_None ? g_backward_workspace_bytes(rows, in, out, N, M, code) : 0);
        void *dy = pointer(dY), *x = pointer(a[1]), *vals = pointer(a[2]), *idx = pointer(a[3]), *w = pointer(ws), *status = pointer(a[13]),
             *stream = handle(a[14]);
        const size_t bytes = (size_t)ws.numel();
        const elsa_status st = unlocked([&] {
            return g_backward(dy, x, rows, vals, (const uint32_t*)idx, out, in, N, M, code, g[0], g[1], g[2], w, bytes, (uint32_t*)status, stream);
        });
        if (st != ELSA_OK) return PyLong_FromLong((long)st);
        PyObject* r = PyTuple_New(3);
        for (int i = 0; r != nullptr && i < 3; ++i) {
            PyObject* t = g[i] != nullptr ? THPVariable_Wrap(grad[i]) : Py_NewRef(Py_None);
            if (t == nullptr) { Py_DECREF(r); return nullptr; }
            PyTuple_SET_ITEM(r, i, t);
        }
        return r;
    });
}

// (vals, idx) of one level, idx None where there are no index words.
PyObject* packed_pair(const at::Tensor& vals, const at::Tensor& idx)
{
    PyObject* v = THPVariable_Wrap(vals);
    PyObject* i = v == nullptr ? nullptr : idx.defined() ? THPVariable_Wrap(idx) : Py_NewRef(Py_None);
    PyObject* r = i == nullptr ? nullptr : PyTuple_Pack(2, v, i);
    Py_XDECREF(v);
    Py_XDECREF(i);
    return r;
}

// W, N, M, dtype code, stream -> (vals, idx)
PyObject* compress(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded(n, 5, [&]() -> PyObject* {
        const at::Tensor& W = matrix(a[0]);
        const int out = (int)size_at(W, 0), in = (int)size_at(W, 1), N = integer(a[1]), M = integer(a[2]);
        const elsa_dtype code = (elsa_dtype)integer(a[3]);
        void *w = pointer(W), *stream = handle(a[4]);
        at::Tensor vals, idx;
        if (g_values_bytes(out, in, N, M, code) != 0) {            // otherwise the entry point says what is wrong
            vals = fresh(W, {out, (int64_t)(in / M) * N}, W.scalar_type());
            const int64_t words = (int64_t)(g_index_bytes(out, in, N, M) / 4);
            if (words > 0) idx = fresh(W, {out, words / out}, at::kInt);
        }
        void *v = vals.defined() ? vals.data_ptr() : nullptr, *i = idx.defined() ? idx.data_ptr() : nullptr;
        const elsa_status st = unlocked([&] { return g_compress(w, out, in, N, M, code, v, (uint32_t*)i, stream); });
        if (st != ELSA_OK) return PyLong_FromLong((long)st);
        return packed_pair(vals, idx);
    });
}

// W, list of N, M, dtype code, stream -> [(vals, idx), ...]; the levels are valid (binding.py checks)
PyObject* compress_levels(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded(n, 5, [&]() -> PyObject* {
        constexpr int kMost = 16;
        const at::Tensor& W = matrix(a[0]);
        const int64_t out = size_at(W, 0), in = size_at(W, 1);
        const int M = integer(a[2]);
        const elsa_dtype code = (elsa_dtype)integer(a[3]);
        if (!PyList_Check(a[1]) || PyList_GET_SIZE(a[1]) > kMost) {
            PyErr_Format(PyExc_ValueError, "a list of at most %d levels expected", kMost);
            throw Raised();
        }
        const int levels = (int)PyList_GET_SIZE(a[1]);
        int N[kMost];
        void* v[kMost];
        uint32_t* x[kMost];
        at::Tensor vals[kMost], idx[kMost];
        for (int l = 0; l < levels; ++l) {
            N[l] = integer(PyList_GET_ITEM(a[1], l));
            vals[l] = fresh(W, {out, in / M * N[l]}, W.scalar_type());
            const int64_t words = (int64_t)(g_index_bytes((int)out, (int)in, N[l], M) / 4);
            if (words > 0) idx[l] = fresh(W, {out, words / out}, at::kInt);
            v[l] = vals[l].data_ptr();
            x[l] = words > 0 ? (uint32_t*)idx[l].data_ptr() : nullptr;
        }
        void *w = pointer(W), *stream = handle(a[4]);
        const elsa_status st = unlocked([&] { return g_compress_levels(w, (int)out, (int)in, M, N, levels, code, v, x, stream); });
        if (st != ELSA_OK) return PyLong_FromLong((long)st);
        PyObject* r = PyList_New(levels);
        for (int l = 0; r != nullptr && l < levels; ++l) {
            PyObject* p = packed_pair(vals[l], idx[l]);
            if (p == nullptr) { Py_DECREF(r); return nullptr; }
            PyList_SET_ITEM(r, l, p);
        }
        return r;
    });
}

// bind({name: address of the entry point})
PyObject* bind(PyObject*, PyObject* table)
{
    auto take = [&](const char* name, auto& f) {
        PyObject* o = PyDict_Check(table) ? PyDict_GetItemString(table, name) : nullptr;
        void* p = o != nullptr ? PyLong_AsVoidPtr(o) : nullptr;
        if (p == nullptr && !PyErr_Occurred()) PyErr_Format(PyExc_KeyError, "no address of %s", name);
        f = reinterpret_cast<std::remove_reference_t<decltype(f)>>(p);
        return p != nullptr;
    };
    const bool ok = take("elsa_nm_linear", g_linear) && take("elsa_nm_linear_masked", g_linear_masked) && take("elsa_nm_linear_i8", g_linear_i8) &&
                    take("elsa_nm_linear_backward", g_backward) && take("elsa_nm_compress", g_compress) &&
                    take("elsa_nm_compress_levels", g_compress_levels) && take("elsa_nm_values_bytes", g_values_bytes) &&
                    take("elsa_nm_index_bytes", g_index_bytes) && take("elsa_workspace_bytes", g_workspace_bytes) &&
                    take("elsa_workspace_bytes_i8", g_workspace_bytes_i8) && take("elsa_backward_workspace_bytes", g_backward_workspace_bytes);
    if (!ok) return nullptr;
    Py_RETURN_NONE;
}

#define ELSA_FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&name)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {ELSA_FAST(linear), ELSA_FAST(linear_masked), ELSA_FAST(linear_i8), ELSA_FAST(linear_backward), ELSA_FAST(compress),
                           ELSA_FAST(compress_levels), {"bind", &bind, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_elsa_host", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

#ifndef ELSA_TORCH_VERSION
#define ELSA_TORCH_VERSION ""
#endif

// torch_version: the torch whose headers this was compiled against; binding.py refuses another.
PyMODINIT_FUNC PyInit__elsa_host()
{
    PyObject* m = PyModule_Create(&g_module);
    if (m != nullptr && PyModule_AddStringConstant(m, "torch_version", ELSA_TORCH_VERSION) != 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
