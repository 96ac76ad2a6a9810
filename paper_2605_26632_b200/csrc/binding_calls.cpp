// The calls of the Python binding that are made once per layer, as plain CPython functions: tensors are read through
// torch's own objects, the result is allocated, and the C ABI is called, without a Python frame or a ctypes object in
// between.  On the smallest layers (7 us of GPU work) the host side is what a caller waits for.
//
// A function takes a call only if every argument has its plain form: tensors of torch's own classes, strided, on CUDA, with
// no wrapper around them (vmap, functionalisation, subclasses), integers as Python ints, no torch-function or
// dispatch mode.  Anything
// else -- wrong types among it -- is answered with None, and the caller (binding.py) takes its general path, which is where
// arguments are refused.  Otherwise the result is what the general path returns, or the library's status as an int.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/core/TensorBody.h>
#include <ATen/ops/empty.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/pybind.h>

#include "../../include/lynx.h"

namespace {

// dense CUDA tensors, with the bookkeeping every one of them carries (autograd, autocast, views)
bool plain_keys(const at::Tensor& t) {
    constexpr c10::DispatchKeySet allowed({c10::DispatchKey::CUDA, c10::DispatchKey::ADInplaceOrView, c10::DispatchKey::AutogradCUDA,
                                           c10::DispatchKey::AutocastCUDA});
    return (t.key_set().raw_repr() & ~allowed.raw_repr()) == 0 && t.has_storage();
}

struct Args {
    bool ok = true;

    const at::Tensor* tensor(PyObject* o) {
        if (!THPVariable_CheckExact(o)) return fail();
        const at::Tensor& t = THPVariable_Unpack(o);
        return t.defined() && plain_keys(t) ? &t : fail();
    }
    const at::Tensor* tensor_or_none(PyObject* o) { return o == Py_None ? nullptr : tensor(o); }
    // 2-D bf16 with unit inner stride
    const at::Tensor* matrix(PyObject* o) {
        const at::Tensor* t = tensor(o);
        return t && t->dim() == 2 && t->scalar_type() == at::kBFloat16 && t->stride(1) == 1 ? t : fail();
    }
    const at::Tensor* two_d(const at::Tensor* t) { return t && t->dim() == 2 ? t : fail(); }
    int64_t integer(PyObject* o) {
        if (!PyLong_CheckExact(o)) return fail(), 0;
        const long long v = PyLong_AsLongLong(o);
        if (v == -1 && PyErr_Occurred()) return PyErr_Clear(), fail(), 0;
        return v;
    }
    lynx_ctx* context(PyObject* o) { return reinterpret_cast<lynx_ctx*>(integer(o)); }

private:
    const at::Tensor* fail() {
        ok = false;
        return nullptr;
    }
};

void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }
template <class T>
T* ptr_as(const at::Tensor* t) { return static_cast<T*>(ptr(t)); }
int64_t ld(const at::Tensor* t) { return t ? t->stride(0) : 0; }
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
at::Tensor empty(at::IntArrayRef shape, const at::Tensor& like, at::ScalarType type = at::kBFloat16) {
    return at::empty(shape, at::TensorOptions().dtype(type).device(like.device()));
}

// What a call returns: `out` as it came in if there was one, else the new tensor.
PyObject* give(PyObject* given, const at::Tensor& made) { return given != Py_None ? Py_NewRef(given) : THPVariable_Wrap(made); }

bool takes(Py_ssize_t nargs, Py_ssize_t want) {
    return nargs == want && !at::impl::torch_function_mode_enabled() && !c10::impl::TorchDispatchModeTLS::any_modes_set();
}

// layer(ctx, X, W, bias, mode, residual, out, fuse)
PyObject* layer(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!takes(n, 8)) Py_RETURN_NONE;
    Args g;
    lynx_ctx* ctx = g.context(a[0]);
    const at::Tensor *X = g.matrix(a[1]), *W = g.matrix(a[2]), *bias = g.tensor_or_none(a[3]), *res = g.tensor_or_none(a[5]);
    const int64_t mode = g.integer(a[4]), fuse = g.integer(a[7]);
    const at::Tensor* out = a[6] == Py_None ? nullptr : g.two_d(g.tensor(a[6]));
    if (res) g.two_d(res);
    if (!g.ok) Py_RETURN_NONE;
    at::Tensor made;
    int s;
    {
        pybind11::gil_scoped_release no_gil;
        const int64_t M = X->size(0), K = X->size(1), N = W->size(0);
        if (!out) out = &(made = empty({M, N}, *X));
        s = lynx_act_sparse_linear(ctx, ptr(X), M, K, ld(X), ptr(W), N, ld(W), ptr(bias), static_cast<lynx_comp_mode>(mode), ptr(res), ld(res),
                                   ptr(out), ld(out), static_cast<lynx_fuse_mode>(fuse), stream());
    }
    return s ? PyLong_FromLong(s) : give(a[6], made);
    END_HANDLE_TH_ERRORS
}

// layer_lora(ctx, X, W, LA, LB, bias, mode, residual, out)
PyObject* layer_lora(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!takes(n, 9)) Py_RETURN_NONE;
    Args g;
    lynx_ctx* ctx = g.context(a[0]);
    const at::Tensor *X = g.matrix(a[1]), *W = g.matrix(a[2]), *LA = g.matrix(a[3]), *LB = g.matrix(a[4]), *bias = g.tensor_or_none(a[5]),
                     *res = g.tensor_or_none(a[7]);
    const int64_t mode = g.integer(a[6]);
    const at::Tensor* out = a[8] == Py_None ? nullptr : g.two_d(g.tensor(a[8]));
    if (res) g.two_d(res);
    if (!g.ok) Py_RETURN_NONE;
    at::Tensor made;
    int s;
    {
        pybind11::gil_scoped_release no_gil;
        const int64_t M = X->size(0), K = X->size(1), N = W->size(0), R = LB->size(0);
        if (!out) out = &(made = empty({M, N}, *X));
        s = lynx_act_sparse_linear_lora(ctx, ptr(X), M, K, ld(X), ptr(W), N, ld(W), ptr(bias), ptr(LA), ld(LA), ptr(LB), ld(LB), R,
                                        static_cast<lynx_comp_mode>(mode), ptr(res), ld(res), ptr(out), ld(out), stream());
    }
    return s ? PyLong_FromLong(s) : give(a[8], made);
    END_HANDLE_TH_ERRORS
}

// layer_fp8(ctx, X, Wq, wscale, bias, mode, residual, out, row_amax)
PyObject* layer_fp8(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!takes(n, 9)) Py_RETURN_NONE;
    Args g;
    lynx_ctx* ctx = g.context(a[0]);
    const at::Tensor *X = g.matrix(a[1]), *Wq = g.two_d(g.tensor(a[2])), *ws = g.tensor_or_none(a[3]), *bias = g.tensor_or_none(a[4]),
                     *res = g.tensor_or_none(a[6]), *amax = g.tensor_or_none(a[8]);
    const int64_t mode = g.integer(a[5]);
    const at::Tensor* out = a[7] == Py_None ? nullptr : g.two_d(g.tensor(a[7]));
    if (res) g.two_d(res);
    if (!g.ok) Py_RETURN_NONE;
    at::Tensor made;
    int s;
    {
        pybind11::gil_scoped_release no_gil;
        const int64_t M = X->size(0), K = X->size(1), N = Wq->size(0);
        if (!out) out = &(made = empty({M, N}, *X));
        s = lynx_act_sparse_linear_fp8(ctx, ptr(X), M, K, ld(X), ptr_as<float>(amax), ptr(Wq), N, ld(Wq), ptr_as<float>(ws), ptr(bias),
                                       static_cast<lynx_comp_mode>(mode), ptr(res), ld(res), ptr(out), ld(out), stream());
    }
    return s ? PyLong_FromLong(s) : give(a[7], made);
    END_HANDLE_TH_ERRORS
}

// prune(ctx, X, mode, values, meta, row_scale) -> (values, meta, row_scale or None)
PyObject* prune(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!takes(n, 6)) Py_RETURN_NONE;
    Args g;
    lynx_ctx* ctx = g.context(a[0]);
    const at::Tensor *X = g.matrix(a[1]), *values = g.tensor_or_none(a[3]), *meta = g.tensor_or_none(a[4]), *scale = g.tensor_or_none(a[5]);
    const int64_t mode = g.integer(a[2]);
    if (!g.ok) Py_RETURN_NONE;
    const bool scaled = mode == LYNX_COMP_ROW || mode == LYNX_COMP_TENSOR;
    at::Tensor v, m, sc;
    int s;
    {
        pybind11::gil_scoped_release no_gil;
        const int64_t M = X->size(0), K = X->size(1);
        if (!values) values = &(v = empty({M, K / 2}, *X));
        if (!meta) meta = &(m = empty({static_cast<int64_t>(lynx_meta_bytes(M, K))}, *X, at::kByte));
        if (!scale && scaled) scale = &(sc = empty({M}, *X, at::kFloat));
        s = lynx_prune_compress(ctx, ptr(X), M, K, ld(X), ptr(values), ptr(meta), ptr_as<float>(scale), static_cast<lynx_comp_mode>(mode),
                                stream());
    }
    if (s) return PyLong_FromLong(s);
    PyObject* t = PyTuple_New(3);
    if (!t) return nullptr;
    PyTuple_SET_ITEM(t, 0, give(a[3], v));
    PyTuple_SET_ITEM(t, 1, give(a[4], m));
    PyTuple_SET_ITEM(t, 2, sc.defined() ? THPVariable_Wrap(sc) : Py_NewRef(a[5]));
    return t;
    END_HANDLE_TH_ERRORS
}

// gemm(ctx, values, meta, W, bias, row_scale, residual, out)
PyObject* gemm(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!takes(n, 8)) Py_RETURN_NONE;
    Args g;
    lynx_ctx* ctx = g.context(a[0]);
    const at::Tensor *values = g.matrix(a[1]), *meta = g.tensor(a[2]), *W = g.matrix(a[3]), *bias = g.tensor_or_none(a[4]),
                     *scale = g.tensor_or_none(a[5]), *res = g.tensor_or_none(a[6]);
    const at::Tensor* out = a[7] == Py_None ? nullptr : g.two_d(g.tensor(a[7]));
    if (res) g.two_d(res);
    if (!g.ok) Py_RETURN_NONE;
    at::Tensor made;
    int s;
    {
        pybind11::gil_scoped_release no_gil;
        const int64_t M = values->size(0), K = values->size(1) * 2, N = W->size(0);
        if (!out) out = &(made = empty({M, N}, *values));
        const lynx_comp comp{ptr_as<float>(scale), ptr(res), ld(res)};
        s = lynx_sparse_linear(ctx, ptr(values), ptr(meta), M, K, ptr(W), N, ld(W), ptr(bias), &comp, ptr(out), ld(out), stream());
    }
    return s ? PyLong_FromLong(s) : give(a[7], made);
    END_HANDLE_TH_ERRORS
}

#define LYNX_FAST(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {LYNX_FAST(layer), LYNX_FAST(layer_lora), LYNX_FAST(layer_fp8), LYNX_FAST(prune), LYNX_FAST(gemm), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_lynx_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__lynx_calls() { return PyModule_Create(&module); }
