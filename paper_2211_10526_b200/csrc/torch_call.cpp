// The call from torch tensors to the C ABI, in C++: checks, strides, output allocation and the current stream.  Small forwards
// are bound by the host, and the same steps as Python attribute look-ups and a ctypes call with thirteen arguments took 12 of
// the 15 microseconds a call cost.  No arithmetic here; the entry points are bound by address, so this module and ctypes use
// one and the same library.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/Functions.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "castling_attn.h"

namespace {

using forward_fn = decltype(&castling_attn_forward);
using strided_fn = decltype(&castling_attn_forward_strided);
forward_fn g_forward = nullptr;
strided_fn g_strided = nullptr;

PyObject* bind(PyObject*, PyObject* args) {
    unsigned long long f = 0, s = 0;
    if (!PyArg_ParseTuple(args, "KK", &f, &s)) return nullptr;
    g_forward = reinterpret_cast<forward_fn>(f);
    g_strided = reinterpret_cast<strided_fn>(s);
    Py_RETURN_NONE;
}

const at::Tensor* tensor(PyObject* o, const char* name) {
    if (THPVariable_Check(o)) return &THPVariable_Unpack(o);
    PyErr_Format(PyExc_TypeError, "%s: expected a torch.Tensor", name);
    return nullptr;
}

PyObject* value_error(const char* what) { PyErr_SetString(PyExc_ValueError, what); return nullptr; }

// forward(handle, ksize, prefix_tokens, q, k, v, dw_weight, dw_bias | None, gridH, gridW, out | None)
// -> the output tensor, or the (non-zero) return code of the C call as an int
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 11 || !g_forward) { PyErr_SetString(PyExc_TypeError, "forward: 11 arguments expected, after bind()"); return nullptr; }
    void* handle = a[0] == Py_None ? nullptr : PyLong_AsVoidPtr(a[0]);
    const long ks = PyLong_AsLong(a[1]), prefix = PyLong_AsLong(a[2]), gridH = PyLong_AsLong(a[8]), gridW = PyLong_AsLong(a[9]);
    if (PyErr_Occurred()) return nullptr;
    const at::Tensor *q = tensor(a[3], "q"), *k = tensor(a[4], "k"), *v = tensor(a[5], "v"), *w = tensor(a[6], "dw_weight");
    const at::Tensor* bias = a[7] == Py_None ? nullptr : tensor(a[7], "dw_bias");
    if (PyErr_Occurred()) return nullptr;
    at::Tensor made;
    const at::Tensor* out = &made;
    if (a[10] == Py_None) made = at::empty_like(*q);
    else if (!(out = tensor(a[10], "out"))) return nullptr;

    if (q->dim() != 4 || k->sizes() != q->sizes() || v->sizes() != q->sizes() || out->sizes() != q->sizes())
        return value_error("q, k, v, out must share one [B, H, N, d] shape");
    const int64_t B = q->size(0), H = q->size(1), N = q->size(2), d = q->size(3);
    if (N != prefix + (int64_t)gridH * gridW) return value_error("N != prefix_tokens + gridH * gridW");
    if (w->dim() != 3 || w->size(0) != H * d || w->size(1) != ks || w->size(2) != ks)
        return value_error("dw_weight must be [H*d, ksize, ksize]");
    const at::ScalarType dt = q->scalar_type();
    if (bias) {
        if (bias->dim() != 1 || bias->size(0) != H * d) return value_error("dw_bias must be [H*d]");
        if (!bias->is_cuda() || !bias->is_contiguous() || bias->scalar_type() != dt)
            return value_error("dw_bias must be a contiguous cuda tensor of the tensors' dtype");
    }
    if (!q->is_cuda() || !k->is_cuda() || !v->is_cuda() || !w->is_cuda() || !out->is_cuda()) return value_error("expected cuda tensors");
    if (!w->is_contiguous()) return value_error("dw_weight must be contiguous");
    const at::Tensor* t[4] = {q, k, v, out};
    const bool contiguous = q->is_contiguous() && k->is_contiguous() && v->is_contiguous() && out->is_contiguous();
    if (!contiguous)
        for (const at::Tensor* x : t)
            if (x->stride(3) != 1) return value_error("the d elements of a token must be contiguous (stride 1 in the last dimension)");
    if (k->scalar_type() != dt || v->scalar_type() != dt || w->scalar_type() != dt || out->scalar_type() != dt) {
        PyErr_SetString(PyExc_TypeError, "all tensors must share one dtype");
        return nullptr;
    }
    if (dt != at::kFloat && dt != at::kBFloat16) {
        PyErr_SetString(PyExc_TypeError, "unsupported dtype: the attention core takes float32 or bfloat16");
        return nullptr;
    }
    if (B > INT32_MAX || H > INT32_MAX || d > INT32_MAX || gridH > INT32_MAX || gridW > INT32_MAX) return value_error("size out of range");
    const castling_dtype_t code = dt == at::kFloat ? CASTLING_F32 : CASTLING_BF16;
    void* stream = c10::cuda::getCurrentCUDAStream(q->get_device()).stream();
    // addresses while the lock is held: a tensor without storage (inside vmap or grad, a fake one) raises here
    const void *qp = q->const_data_ptr(), *kp = k->const_data_ptr(), *vp = v->const_data_ptr(), *wp = w->const_data_ptr();
    const void* bp = bias ? bias->const_data_ptr() : nullptr;
    void* op = out->mutable_data_ptr();
    int rc;
    PyThreadState* gil = PyEval_SaveThread();   // a first call of a larger shape allocates and waits for the device
    if (contiguous) {
        rc = g_forward(static_cast<castling_attn_t*>(handle), qp, kp, vp, wp, bp, op, (int)B, (int)H, (int)gridH, (int)gridW, (int)d,
                       code, stream);
    } else {   // views of token-major or fused-projection buffers: pass their strides through
        long long s[12];
        for (int i = 0; i < 4; ++i)
            for (int j = 0; j < 3; ++j) s[3 * i + j] = t[i]->stride(j);
        const castling_attn_layout_t layout = {s[0], s[1], s[2], s[3], s[4], s[5], s[6], s[7], s[8], s[9], s[10], s[11]};
        rc = g_strided(static_cast<castling_attn_t*>(handle), qp, kp, vp, wp, bp, op, (int)B, (int)H, (int)gridH, (int)gridW, (int)d,
                       code, &layout, stream);
    }
    PyEval_RestoreThread(gil);
    if (rc != CASTLING_OK) return PyLong_FromLong(rc);
    if (a[10] != Py_None) { Py_INCREF(a[10]); return a[10]; }
    return THPVariable_Wrap(std::move(made));
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, "bind(address of castling_attn_forward, address of castling_attn_forward_strided)"},
    {"forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(forward)), METH_FASTCALL, "one forward on torch tensors"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_torch_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__torch_call() {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_against", BUILT_AGAINST) != 0) { Py_DECREF(m); return nullptr; }
    return m;
}
