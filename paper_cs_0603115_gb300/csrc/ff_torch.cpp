// ff_torch.cpp -- native front of the Python wrappers: argument checks, output
// allocation, workspace lookup, current stream and the call of the C ABI in one
// step, for the calls the wrappers spend most on.  On short vectors the kernel
// takes 2-5 us and the wrapper, in Python alone, 16-24 (ff.add 16.2 us a call,
// ff.dot 18.6, ff.gemv_t 23.6), so such calls are host bound; through this front
// they take 4.0, 4.2 and 4.1, of which 1.3 is the output's allocation.
//
// Every function takes the address of its C entry point first and does the
// call only when all arguments pass the checks the Python wrapper makes (and
// no tensor subclass, functional transform or dispatch mode is involved);
// otherwise it returns None without having done anything, and the wrapper
// takes its own path, which raises the error or serves the case.  It returns
// the output tensor(s), or the status code of a call that failed.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/ff.h"

namespace {

// The current device and stream of one call.
struct Where {
    c10::DeviceIndex dev;
    cudaStream_t stream;
};

// `first`: an argument; without a plain CUDA tensor there the device is not asked.
bool where(PyObject* first, Where* w)
{
    if (!THPVariable_CheckExact(first) || !THPVariable_Unpack(first).is_cuda()) return false;
    // modes see every tensor operation of the Python path
    if (at::impl::torch_function_mode_enabled() || c10::impl::TorchDispatchModeTLS::any_modes_set()) return false;
    w->dev = c10::cuda::current_device();
    w->stream = c10::cuda::getCurrentCUDAStream(w->dev).stream();
    return true;
}

// A plain contiguous float32 CUDA tensor on the current device.
const at::Tensor* plain(PyObject* o, const Where& w)
{
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || t.scalar_type() != at::kFloat || t.layout() != at::kStrided) return nullptr;
    const c10::DispatchKeySet ks = t.key_set();
    if (ks.has(c10::DispatchKey::Python) || ks.has(c10::DispatchKey::FuncTorchBatched) ||
        ks.has(c10::DispatchKey::FuncTorchGradWrapper) || ks.has(c10::DispatchKey::Functionalize))
        return nullptr;
    if (!t.unsafeGetTensorImpl()->has_storage() || t.get_device() != w.dev || !t.is_contiguous()) return nullptr;
    return &t;
}

// The same with a last dimension of two.
const at::Tensor* pairs(PyObject* o, const Where& w)
{
    const at::Tensor* t = plain(o, w);
    return t != nullptr && t->dim() >= 1 && t->size(-1) == 2 ? t : nullptr;
}

const ff2* in(const at::Tensor& t) { return static_cast<const ff2*>(t.data_ptr()); }
ff2* out(const at::Tensor& t) { return static_cast<ff2*>(t.data_ptr()); }
size_t values(const at::Tensor& t) { return static_cast<size_t>(t.numel()) / 2; }

template <class F>
F entry(PyObject* address)
{
    return reinterpret_cast<F>(PyLong_AsVoidPtr(address));
}

// The caller's output (checked against `sizes`) or a new one like `like`.
bool output(PyObject* o, at::IntArrayRef sizes, const at::Tensor& like, const Where& w, at::Tensor* t)
{
    if (o == Py_None) {
        *t = at::empty(sizes, like.options());
        return true;
    }
    const at::Tensor* g = plain(o, w);
    if (g == nullptr || g->sizes() != sizes) return false;
    *t = *g;
    return true;
}

PyObject* wrap(PyObject* given, const at::Tensor& t)
{
    if (given != Py_None) {
        Py_INCREF(given);
        return given;
    }
    return THPVariable_Wrap(t);
}

size_t held(const at::Tensor& ws) { return static_cast<size_t>(ws.numel()); }

// The wrapper's cached workspace of this device, stream and key (a reference of
// its own: another thread may clear the cache during the call), if it holds
// `bytes`.
bool workspace(PyObject* cache, PyObject* key, const Where& w, size_t bytes, at::Tensor* ws)
{
    PyObject* k = Py_BuildValue("(iKO)", static_cast<int>(w.dev), reinterpret_cast<unsigned long long>(w.stream), key);
    if (k == nullptr) return false;
    PyObject* o = PyDict_GetItemWithError(cache, k);   // borrowed
    Py_DECREF(k);
    if (o == nullptr || !THPVariable_CheckExact(o)) return false;
    *ws = THPVariable_Unpack(o);
    return held(*ws) >= bytes;
}

// The call with the GIL released, as a ctypes call makes it; held again when the
// call throws too, since what becomes of the exception touches Python.
template <class Call>
ff_status unlocked(Call&& call)
{
    struct Released {
        PyThreadState* state = PyEval_SaveThread();
        ~Released() { PyEval_RestoreThread(state); }
    } released;
    return call();
}

// nullptr from the body means "not taken": None.  C++ exceptions (an allocation
// that fails, say) become the Python ones torch raises.
template <class Body>
PyObject* guarded(Body&& body)
{
    HANDLE_TH_ERRORS
    PyObject* r = body();
    if (r == nullptr && !PyErr_Occurred()) Py_RETURN_NONE;
    return r;
    END_HANDLE_TH_ERRORS
}

using Unary = ff_status (*)(const ff2*, ff2*, size_t, cudaStream_t);
using Binary = ff_status (*)(const ff2*, const ff2*, ff2*, size_t, cudaStream_t);

PyObject* status(ff_status st) { return PyLong_FromLong(static_cast<long>(st)); }

// unary(address, x, out)
PyObject* unary(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        Where w;
        if (n != 3 || !where(a[1], &w)) return nullptr;
        const at::Tensor* x = pairs(a[1], w);
        at::Tensor o;
        if (!x || !output(a[2], x->sizes(), *x, w, &o)) return nullptr;
        const auto f = entry<Unary>(a[0]);
        const ff_status st = unlocked([&] { return f(in(*x), out(o), values(*x), w.stream); });
        return st == FF_OK ? wrap(a[2], o) : status(st);
    });
}

// binary(address, a, b, out)
PyObject* binary(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        Where w;
        if (n != 4 || !where(a[1], &w)) return nullptr;
        const at::Tensor *x = pairs(a[1], w), *y = pairs(a[2], w);
        at::Tensor o;
        if (!x || !y || x->sizes() != y->sizes() || !output(a[3], x->sizes(), *x, w, &o)) return nullptr;
        const auto f = entry<Binary>(a[0]);
        const ff_status st = unlocked([&] { return f(in(*x), in(*y), out(o), values(*x), w.stream); });
        return st == FF_OK ? wrap(a[3], o) : status(st);
    });
}

// axpy(address, hi, lo, x, y, out)
PyObject* axpy(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        Where w;
        if (n != 6 || !PyFloat_CheckExact(a[1]) || !PyFloat_CheckExact(a[2]) || !where(a[3], &w)) return nullptr;
        const at::Tensor *x = pairs(a[3], w), *y = pairs(a[4], w);
        at::Tensor o;
        if (!x || !y || x->sizes() != y->sizes() || !output(a[5], x->sizes(), *x, w, &o)) return nullptr;
        const ff2 alpha = {static_cast<float>(PyFloat_AS_DOUBLE(a[1])), static_cast<float>(PyFloat_AS_DOUBLE(a[2]))};
        const auto f = entry<decltype(&ff_axpy)>(a[0]);
        const ff_status st = unlocked([&] { return f(alpha, in(*x), in(*y), out(o), values(*x), w.stream); });
        return st == FF_OK ? wrap(a[5], o) : status(st);
    });
}

// reduce1(address, x, out, ff values, address of the workspace size, cache, key): ff_sum
// (float-float values) and ff_sum2 (binary32 values)
PyObject* reduce1(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        Where w;
        if (n != 7 || !where(a[1], &w)) return nullptr;
        const bool ff = a[3] == Py_True;
        const at::Tensor* x = ff ? pairs(a[1], w) : plain(a[1], w);
        if (!x) return nullptr;
        const size_t len = ff ? values(*x) : static_cast<size_t>(x->numel());
        at::Tensor ws;
        if (!workspace(a[5], a[6], w, entry<decltype(&ff_reduce_workspace_bytes)>(a[4])(len), &ws)) return nullptr;
        at::Tensor o;
        if (!output(a[2], {2}, *x, w, &o)) return nullptr;
        const auto f = entry<ff_status (*)(const void*, size_t, ff2*, void*, size_t, cudaStream_t)>(a[0]);
        const ff_status st =
            unlocked([&] { return f(x->data_ptr(), len, out(o), ws.data_ptr(), held(ws), w.stream); });
        return st == FF_OK ? wrap(a[2], o) : status(st);
    });
}

// reduce2(address, x, y, out, ff values, address of the workspace size, cache, key): ff_dot,
// ff_dot2
PyObject* reduce2(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        Where w;
        if (n != 8 || !where(a[1], &w)) return nullptr;
        const bool ff = a[4] == Py_True;
        const at::Tensor* x = ff ? pairs(a[1], w) : plain(a[1], w);
        const at::Tensor* y = ff ? pairs(a[2], w) : plain(a[2], w);
        if (!x || !y || (ff ? x->sizes() != y->sizes() : x->numel() != y->numel())) return nullptr;
        const size_t len = ff ? values(*x) : static_cast<size_t>(x->numel());
        at::Tensor ws;
        if (!workspace(a[6], a[7], w, entry<decltype(&ff_reduce_workspace_bytes)>(a[5])(len), &ws)) return nullptr;
        at::Tensor o;
        if (!output(a[3], {2}, *x, w, &o)) return nullptr;
        const auto f = entry<ff_status (*)(const void*, const void*, size_t, ff2*, void*, size_t, cudaStream_t)>(a[0]);
        const ff_status st =
            unlocked([&] { return f(x->data_ptr(), y->data_ptr(), len, out(o), ws.data_ptr(), held(ws), w.stream); });
        return st == FF_OK ? wrap(a[3], o) : status(st);
    });
}

// dot_backward(address, dout, x, y, dx, dy) -> (dx, dy)
PyObject* dot_backward(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject* {
        Where w;
        if (n != 6 || !where(a[1], &w)) return nullptr;
        const at::Tensor *d = pairs(a[1], w), *x = pairs(a[2], w), *y = pairs(a[3], w);
        at::Tensor dx, dy;
        if (!d || !x || !y || d->numel() != 2 || x->sizes() != y->sizes() || !output(a[4], x->sizes(), *x, w, &dx) ||
            !output(a[5], y->sizes(), *y, w, &dy))
            return nullptr;
        const auto f = entry<decltype(&ff_dot_backward)>(a[0]);
        const ff_status st =
            unlocked([&] { return f(in(*d), in(*x), in(*y), out(dx), out(dy), values(*x), w.stream); });
        if (st != FF_OK) return status(st);
        PyObject* px = wrap(a[4], dx);
        PyObject* py = px ? wrap(a[5], dy) : nullptr;
        PyObject* r = py ? PyTuple_Pack(2, px, py) : nullptr;
        Py_XDECREF(px);
        Py_XDECREF(py);
        return r;
    });
}

// gemv(address, A, X, out): Y = A X
PyObject* gemv(PyObject*, PyObject* const* a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        Where w;
        if (na != 4 || !where(a[1], &w)) return nullptr;
        const at::Tensor *A = pairs(a[1], w), *X = pairs(a[2], w);
        if (!A || !X || A->dim() != 3 || X->dim() != 3 || X->size(1) != A->size(1)) return nullptr;
        const int64_t m = A->size(0), n = A->size(1), k = X->size(0);
        at::Tensor o;
        if (!output(a[3], {k, m, 2}, *A, w, &o)) return nullptr;
        const auto f = entry<decltype(&ff_gemv)>(a[0]);
        const ff_status st = unlocked([&] { return f(in(*A), m, n, n, in(*X), n, k, out(o), m, w.stream); });
        return st == FF_OK ? wrap(a[3], o) : status(st);
    });
}

// gemv_t(address, A, dY, out, address of the workspace size, cache, key)
PyObject* gemv_t(PyObject*, PyObject* const* a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        Where w;
        if (na != 7 || !where(a[1], &w)) return nullptr;
        const at::Tensor *A = pairs(a[1], w), *dY = pairs(a[2], w);
        if (!A || !dY || A->dim() != 3 || dY->dim() != 3 || dY->size(1) != A->size(0)) return nullptr;
        const int64_t m = A->size(0), n = A->size(1), k = dY->size(0);
        at::Tensor ws;
        if (!workspace(a[5], a[6], w, entry<decltype(&ff_gemv_t_workspace_bytes)>(a[4])(m, n, k), &ws)) return nullptr;
        at::Tensor o;
        if (!output(a[3], {k, n, 2}, *A, w, &o)) return nullptr;
        const auto f = entry<decltype(&ff_gemv_t)>(a[0]);
        const ff_status st =
            unlocked([&] { return f(in(*A), m, n, n, in(*dY), m, k, out(o), n, ws.data_ptr(), held(ws), w.stream); });
        return st == FF_OK ? wrap(a[3], o) : status(st);
    });
}

// gemv_dA(address, dY, X, out)
PyObject* gemv_dA(PyObject*, PyObject* const* a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        Where w;
        if (na != 4 || !where(a[1], &w)) return nullptr;
        const at::Tensor *dY = pairs(a[1], w), *X = pairs(a[2], w);
        if (!dY || !X || dY->dim() != 3 || X->dim() != 3 || dY->size(0) != X->size(0)) return nullptr;
        const int64_t k = dY->size(0), m = dY->size(1), n = X->size(1);
        at::Tensor o;
        if (!output(a[3], {m, n, 2}, *dY, w, &o)) return nullptr;
        const auto f = entry<decltype(&ff_gemv_dA)>(a[0]);
        const ff_status st = unlocked([&] { return f(in(*dY), m, m, in(*X), n, n, k, out(o), n, w.stream); });
        return st == FF_OK ? wrap(a[3], o) : status(st);
    });
}

// gemm(address, A, B, transa, transb, out)
PyObject* gemm(PyObject*, PyObject* const* a, Py_ssize_t na)
{
    return guarded([&]() -> PyObject* {
        Where w;
        if (na != 6 || !PyBool_Check(a[3]) || !PyBool_Check(a[4]) || !where(a[1], &w)) return nullptr;
        const bool ta = a[3] == Py_True, tb = a[4] == Py_True;
        const at::Tensor *A = pairs(a[1], w), *B = pairs(a[2], w);
        if (!A || !B || A->dim() != 3 || B->dim() != 3) return nullptr;
        const int64_t k = A->size(ta ? 0 : 1), m = A->size(ta ? 1 : 0);
        const int64_t n = B->size(tb ? 0 : 1);
        if (B->size(tb ? 1 : 0) != k) return nullptr;
        at::Tensor o;
        if (!output(a[5], {m, n, 2}, *A, w, &o)) return nullptr;
        const int64_t lda = std::max<int64_t>(A->size(1), 1), ldb = std::max<int64_t>(B->size(1), 1);
        const auto f = entry<decltype(&ff_gemm)>(a[0]);
        const ff_status st = unlocked([&] {
            return f(ta, tb, m, n, k, in(*A), lda, in(*B), ldb, out(o), std::max<int64_t>(n, 1), w.stream);
        });
        return st == FF_OK ? wrap(a[5], o) : status(st);
    });
}

#define FF_METHOD(name) \
    {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FF_METHOD(unary),        FF_METHOD(binary), FF_METHOD(axpy),    FF_METHOD(reduce1), FF_METHOD(reduce2),
                         FF_METHOD(dot_backward), FF_METHOD(gemv),   FF_METHOD(gemv_t), FF_METHOD(gemv_dA), FF_METHOD(gemm),
                         {nullptr, nullptr, 0, nullptr}};

PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_ffnative", "Native front of the wrappers.", -1, methods,
                          nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__ffnative(void) { return PyModule_Create(&module_def); }
