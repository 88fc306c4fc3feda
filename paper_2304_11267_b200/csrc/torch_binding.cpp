// CPython extension `_sd_torch`: the calls of binding.py on torch tensors, marshalled without the interpreter.
//
// A small call of a UNet step keeps the GPU busy for 4-6 us, less than ctypes needs to marshal it: reading four
// tensors' attributes, asking for the stream, allocating the result and converting thirteen arguments in Python took
// 11 us a call (attention 64 tokens, d = 160), 13 us with three more tensors (group normalisation).  Here the same
// checks are member reads of the C++ tensors, the result comes straight from the caching allocator and the C ABI is
// called directly.  Errors of the C ABI are returned as its integer status (binding.py raises them, and lends the
// two-pass workspace where that is what is missing); bad tensors raise here.
#include <Python.h>

#include <cmath>

#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/sd_attn.h"
#include "../../include/sd_geglu.h"
#include "../../include/sd_groupnorm.h"
#include "../../include/sd_winograd.h"

namespace {

using at::Tensor;

// The tensor behind a Python object; nullptr with a Python error set where it is none.
const Tensor* tensor_of(PyObject* o, const char* what) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a torch tensor", what);
        return nullptr;
    }
    return &THPVariable_Unpack(o);
}

bool stream_of(PyObject* o, const Tensor& on, void** stream) {
    if (o == Py_None) {
        *stream = c10::cuda::getCurrentCUDAStream(on.device().index()).stream();
        return true;
    }
    *stream = PyLong_AsVoidPtr(o);
    return !(*stream == nullptr && PyErr_Occurred());
}

int dtype_code(const Tensor& t) {
    switch (t.scalar_type()) {
        case at::kHalf: return SD_ATTN_F16;
        case at::kFloat: return SD_ATTN_F32;
        case at::kBFloat16: return SD_ATTN_BF16;
        default: return -1;
    }
}

Tensor empty_on(const Tensor& like, at::IntArrayRef sizes) {
    return at::detail::empty_cuda(sizes, like.scalar_type(), like.device(), std::nullopt);
}

// Lets other Python threads run: an allocation may wait for the device, and a launch waits where its queue is full -- perhaps for
// a host function that itself needs the interpreter.  No Python call inside.
struct OtherThreadsRun {
    PyThreadState* state = PyEval_SaveThread();
    ~OtherThreadsRun() { PyEval_RestoreThread(state); }
};

// The result object: the caller's `out` where one was given, else the new tensor.
PyObject* result(PyObject* out, Tensor&& made) {
    if (out == Py_None) return THPVariable_Wrap(std::move(made));
    Py_INCREF(out);
    return out;
}

// attention(handle, layout, q, k, v, scale or None, out or None, stream or None) -> out, or an int status
PyObject* attention_impl(PyObject* const* a) {
    auto* h = a[0] == Py_None ? nullptr : (sd_attn_handle*)PyLong_AsVoidPtr(a[0]);   // None: a closed handle
    const long layout = PyLong_AsLong(a[1]);
    if (PyErr_Occurred()) return nullptr;
    const Tensor *q = tensor_of(a[2], "q"), *k = q ? tensor_of(a[3], "k") : nullptr, *v = k ? tensor_of(a[4], "v") : nullptr;
    if (!v) return nullptr;
    if (!(q->is_cuda() && k->is_cuda() && v->is_cuda())) {
        PyErr_SetString(PyExc_ValueError, "q, k, v must be CUDA tensors");
        return nullptr;
    }
    if (!(q->is_contiguous() && k->is_contiguous() && v->is_contiguous())) {
        PyErr_SetString(PyExc_ValueError, "q, k, v must be contiguous [B,H,N,d] (or, token-major, [B,N,H,d]) tensors");
        return nullptr;
    }
    const int dtype = dtype_code(*q);
    if (dtype < 0) {
        PyErr_SetString(PyExc_TypeError, "float16, bfloat16 or float32 only");
        return nullptr;
    }
    if (q->dim() != 4 || k->dim() != 4) {
        PyErr_SetString(PyExc_ValueError, "q and k must have four dimensions");
        return nullptr;
    }
    const bool tokens_first = layout == SD_ATTN_LAYOUT_BNHD;
    const at::IntArrayRef s = q->sizes();
    const int64_t H = s[tokens_first ? 2 : 1], Nq = s[tokens_first ? 1 : 2], Nk = k->size(tokens_first ? 1 : 2), d = s[3];
    double scale = 1.0;
    if (a[5] == Py_None) {
        scale = std::pow((double)d, -0.5);
    } else {
        scale = PyFloat_AsDouble(a[5]);
        if (scale == -1.0 && PyErr_Occurred()) return nullptr;
    }
    void* stream;
    if (!stream_of(a[7], *q, &stream)) return nullptr;
    Tensor made;
    const Tensor* out = &made;
    if (a[6] != Py_None && !(out = tensor_of(a[6], "out"))) return nullptr;
    int rc;
    {
        OtherThreadsRun scope;
        if (out == &made) made = empty_on(*q, s);
        rc = sd_attn_forward(h, q->data_ptr(), k->data_ptr(), v->data_ptr(), out->data_ptr(), (int)s[0], (int)H, (int)Nq, (int)Nk,
                             (int)d, (float)scale, dtype, stream);
    }
    if (rc != SD_ATTN_OK) return PyLong_FromLong(rc);
    return result(a[6], std::move(made));
}

// geglu(x, out or None, stream or None) -> out, or an int status
PyObject* geglu_impl(PyObject* const* a) {
    const Tensor* x = tensor_of(a[0], "x");
    if (!x) return nullptr;
    if (!x->is_cuda() || !x->is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "x must be a contiguous CUDA tensor");
        return nullptr;
    }
    const int dtype = dtype_code(*x);
    const int64_t dim = x->dim(), last = dim > 0 ? x->size(dim - 1) : 1;
    if ((dtype != SD_ATTN_F16 && dtype != SD_ATTN_F32) || last % 2) {
        PyErr_SetString(PyExc_ValueError, "x must be float16 or float32 with an even last dimension");
        return nullptr;
    }
    const int64_t C = last / 2, rows = C ? x->numel() / last : 0;
    void* stream;
    if (!stream_of(a[2], *x, &stream)) return nullptr;
    Tensor made;
    const Tensor* out = &made;
    if (a[1] != Py_None && !(out = tensor_of(a[1], "out"))) return nullptr;
    int rc;
    {
        OtherThreadsRun scope;
        if (out == &made) {
            c10::SmallVector<int64_t, 5> sizes(x->sizes().begin(), x->sizes().end());
            sizes[dim - 1] = C;
            made = empty_on(*x, sizes);
        }
        rc = sd_geglu_forward(x->data_ptr(), out->data_ptr(), rows, (int)C, dtype, stream);
    }
    if (rc != SD_ATTN_OK) return PyLong_FromLong(rc);
    return result(a[1], std::move(made));
}

// groupnorm(x, groups, eps, gamma or None, beta or None, out or None, stream or None) -> out, or an int status
PyObject* groupnorm_impl(PyObject* const* a) {
    const Tensor* x = tensor_of(a[0], "x");
    if (!x) return nullptr;
    if (!x->is_cuda() || !x->is_contiguous() || x->dim() < 2) {
        PyErr_SetString(PyExc_ValueError, "x must be a contiguous CUDA tensor [N, C, ...]");
        return nullptr;
    }
    const int dtype = dtype_code(*x);
    if (dtype != SD_ATTN_F16 && dtype != SD_ATTN_F32) {
        PyErr_SetString(PyExc_ValueError, "x must be float16 or float32");
        return nullptr;
    }
    const int64_t N = x->size(0), C = x->size(1), HW = N * C ? x->numel() / (N * C) : 1;
    const long groups = PyLong_AsLong(a[1]);
    if (groups == -1 && PyErr_Occurred()) return nullptr;
    const double eps = PyFloat_AsDouble(a[2]);
    if (eps == -1.0 && PyErr_Occurred()) return nullptr;
    const void* affine[2] = {nullptr, nullptr};
    for (int i = 0; i < 2; ++i) {
        if (a[3 + i] == Py_None) continue;
        const Tensor* t = tensor_of(a[3 + i], i ? "beta" : "gamma");
        if (!t) return nullptr;
        if (t->scalar_type() != x->scalar_type() || t->dim() != 1 || t->size(0) != C || !t->is_cuda() || !t->is_contiguous()) {
            PyErr_SetString(PyExc_ValueError, "gamma and beta must be contiguous CUDA tensors [C] of x's dtype");
            return nullptr;
        }
        affine[i] = t->data_ptr();
    }
    void* stream;
    if (!stream_of(a[6], *x, &stream)) return nullptr;
    Tensor made;
    const Tensor* out = &made;
    if (a[5] != Py_None && !(out = tensor_of(a[5], "out"))) return nullptr;
    int rc;
    {
        OtherThreadsRun scope;
        if (out == &made) made = empty_on(*x, x->sizes());
        rc = sd_groupnorm_forward(x->data_ptr(), affine[0], affine[1], out->data_ptr(), (int)N, (int)C, HW, (int)groups, (float)eps, dtype,
                                  stream);
    }
    if (rc != SD_ATTN_OK) return PyLong_FromLong(rc);
    return result(a[5], std::move(made));
}

// conv3x3(x, packed filter, bias or None, K, C, out or None, stream or None) -> out, or an int status
PyObject* conv3x3_impl(PyObject* const* a) {
    const Tensor *x = tensor_of(a[0], "x"), *packed = x ? tensor_of(a[1], "packed") : nullptr;
    if (!packed) return nullptr;
    const Tensor* bias = nullptr;
    if (a[2] != Py_None && !(bias = tensor_of(a[2], "bias"))) return nullptr;
    const long K = PyLong_AsLong(a[3]), C = PyLong_AsLong(a[4]);
    if (PyErr_Occurred()) return nullptr;
    if (!x->is_cuda() || x->scalar_type() != at::kHalf || !x->is_contiguous() || x->dim() != 4 || x->size(3) != C) {
        PyErr_Format(PyExc_ValueError, "x must be a contiguous float16 CUDA tensor [N,H,W,%ld]", C);
        return nullptr;
    }
    const int64_t N = x->size(0), H = x->size(1), W = x->size(2);
    void* stream;
    if (!stream_of(a[6], *x, &stream)) return nullptr;
    Tensor made;
    const Tensor* out = &made;
    if (a[5] != Py_None && !(out = tensor_of(a[5], "out"))) return nullptr;
    int rc;
    {
        OtherThreadsRun scope;
        const int preferred = N == 0 ? 1 : sd_winograd_direct_preferred((int)N, (int)H, (int)W, (int)C, (int)K);
        rc = preferred < 0 ? -preferred : SD_ATTN_ERR_UNSUPPORTED;
        if (preferred > 0) {
            if (out == &made) made = empty_on(*x, {N, H, W, (int64_t)K});
            rc = sd_winograd_direct_forward(x->data_ptr(), packed->data_ptr(), bias ? bias->data_ptr() : nullptr, out->data_ptr(), (int)N,
                                            (int)H, (int)W, (int)C, (int)K, stream);
        }
    }
    if (rc != SD_ATTN_OK) return PyLong_FromLong(rc);
    return result(a[5], std::move(made));
}

// A C++ exception (out of memory in the caching allocator, say) becomes the Python error torch itself would raise.
template <PyObject* (*IMPL)(PyObject* const*), int N_ARGS>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != N_ARGS) {
        PyErr_Format(PyExc_TypeError, "%d arguments expected, %zd given", N_ARGS, n);
        return nullptr;
    }
    HANDLE_TH_ERRORS
    return IMPL(args);
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"attention", (PyCFunction)(void*)entry<attention_impl, 8>, METH_FASTCALL, "sd_attn_forward on torch tensors"},
    {"geglu", (PyCFunction)(void*)entry<geglu_impl, 3>, METH_FASTCALL, "sd_geglu_forward on torch tensors"},
    {"groupnorm", (PyCFunction)(void*)entry<groupnorm_impl, 7>, METH_FASTCALL, "sd_groupnorm_forward on torch tensors"},
    {"conv3x3", (PyCFunction)(void*)entry<conv3x3_impl, 7>, METH_FASTCALL, "sd_winograd_direct_forward on torch tensors"},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_sd_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__sd_torch() { return PyModule_Create(&module); }
