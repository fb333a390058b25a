// The forward entry points as a CPython extension over torch tensors: what binding.py does for a call - output allocation, data
// pointers, current stream, the call into libboda.so without the GIL - in native code.
//
// Bound: the host.  A small layer's kernel takes 2 to 7 us, and the interpreter with ctypes took 6.7 us a call; this takes 3.8 to 4.2, of which
// 2.3 are the launch itself.
// Only the ordinary call is taken here (plain CUDA tensors, current stream); every function returns None for anything else, before it
// has done anything, and the caller goes on through ctypes.  A status other than 0 is returned as an int.
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>

#include "boda.h"

namespace {

decltype(&boda_conv_fwd_planned) g_planned = nullptr;
decltype(&boda_conv_fwd) g_forward = nullptr;
decltype(&boda_sgemm) g_sgemm = nullptr;
decltype(&boda_conv_out_dim) g_out_dim = nullptr;

// A plain tensor (or parameter) with CUDA memory of its own.
const at::Tensor* plain(PyObject* o)
{
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    return t.defined() && t.is_cuda() && t.layout() == at::kStrided ? &t : nullptr;
}

// nullptr in `t` for None; false if the argument is neither None nor a plain tensor
bool optional(PyObject* o, const at::Tensor** t)
{
    *t = nullptr;
    return o == Py_None || (*t = plain(o)) != nullptr;
}

bool small_int(PyObject* o, int* v)
{
    if (!PyLong_CheckExact(o)) return false;
    int overflow = 0;
    const long l = PyLong_AsLongAndOverflow(o, &overflow);
    if (overflow || l < INT_MIN || l > INT_MAX) return false;
    *v = (int)l;
    return true;
}

float* data(const at::Tensor* t) { return t ? static_cast<float*>(t->mutable_data_ptr()) : nullptr; }
void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
struct NoGil {
    PyThreadState* state = PyEval_SaveThread();
    ~NoGil() { PyEval_RestoreThread(state); }
};

// planned(handle, workspace, out_shape, x, filt, bias, out)
PyObject* planned(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    const at::Tensor *ws, *x, *filt, *bias, *out;
    if (n != 7 || !PyLong_CheckExact(a[0]) || !optional(a[1], &ws) || !PyTuple_CheckExact(a[2]) || PyTuple_GET_SIZE(a[2]) != 4 ||
        !(x = plain(a[3])) || !(filt = plain(a[4])) || !optional(a[5], &bias) || !optional(a[6], &out) || at::impl::torch_function_mode_enabled())
        Py_RETURN_NONE;
    auto* handle = static_cast<boda_conv_plan*>(PyLong_AsVoidPtr(a[0]));
    if (PyErr_Occurred()) { PyErr_Clear(); Py_RETURN_NONE; }
    at::Tensor fresh;
    int64_t shape[4] = {0, 0, 0, 0};
    if (!out) {
        if (x->scalar_type() != at::kFloat) Py_RETURN_NONE;
        for (int i = 0; i < 4; ++i) {
            int v;
            if (!small_int(PyTuple_GET_ITEM(a[2], i), &v)) Py_RETURN_NONE;
            shape[i] = v;
        }
    }
    int status;
    {
        NoGil nogil;
        if (!out) fresh = x->new_empty(shape);
        status = g_planned(handle, data(x), data(filt), data(bias), data(out ? out : &fresh), data(ws), current_stream());
    }
    if (status != 0) return PyLong_FromLong(status);
    return out ? Py_NewRef(a[6]) : THPVariable_Wrap(std::move(fresh));
    END_HANDLE_TH_ERRORS
}

// conv_fwd(x, filt, bias, stride, pad, relu)
PyObject* conv_fwd(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    const at::Tensor *x, *filt, *bias;
    int stride, pad;
    if (n != 6 || !(x = plain(a[0])) || !(filt = plain(a[1])) || !optional(a[2], &bias) || !small_int(a[3], &stride) || !small_int(a[4], &pad) ||
        x->dim() != 4 || filt->dim() != 4 || x->scalar_type() != at::kFloat || at::impl::torch_function_mode_enabled())
        Py_RETURN_NONE;
    const int relu = PyObject_IsTrue(a[5]);
    if (relu < 0) return nullptr;
    int d[7];
    const int64_t sizes[7] = {x->size(0), x->size(1), x->size(2), x->size(3), filt->size(0), filt->size(2), filt->size(3)};
    for (int i = 0; i < 7; ++i) {
        if (sizes[i] > INT_MAX) Py_RETURN_NONE;
        d[i] = (int)sizes[i];
    }
    const int64_t shape[4] = {d[0], d[4], g_out_dim(d[2], d[5], stride, pad), g_out_dim(d[3], d[6], stride, pad)};
    at::Tensor out;
    int status;
    {
        NoGil nogil;
        out = x->new_empty(shape);
        status = g_forward(data(x), data(filt), data(bias), data(&out), d[0], d[1], d[2], d[3], d[4], d[5], d[6], stride, pad, relu, current_stream());
    }
    return status != 0 ? PyLong_FromLong(status) : THPVariable_Wrap(std::move(out));
    END_HANDLE_TH_ERRORS
}

// sgemm(A, B, C, M, N, K) -> status
PyObject* sgemm(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    const at::Tensor *A, *B, *C;
    int m[3];
    if (n != 6 || !(A = plain(a[0])) || !(B = plain(a[1])) || !(C = plain(a[2])) || !small_int(a[3], &m[0]) || !small_int(a[4], &m[1]) ||
        !small_int(a[5], &m[2]) || at::impl::torch_function_mode_enabled())
        Py_RETURN_NONE;
    int status;
    {
        NoGil nogil;
        status = g_sgemm(data(A), data(B), data(C), m[0], m[1], m[2], current_stream());
    }
    return PyLong_FromLong(status);
    END_HANDLE_TH_ERRORS
}

// bind(boda_conv_fwd_planned, boda_conv_fwd, boda_sgemm, boda_conv_out_dim): addresses of the entry points
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 4) { PyErr_SetString(PyExc_TypeError, "bind takes four addresses"); return nullptr; }
    void* p[4];
    for (int i = 0; i < 4; ++i) {
        p[i] = PyLong_AsVoidPtr(a[i]);
        if (PyErr_Occurred()) return nullptr;
    }
    g_planned = reinterpret_cast<decltype(g_planned)>(p[0]);
    g_forward = reinterpret_cast<decltype(g_forward)>(p[1]);
    g_sgemm = reinterpret_cast<decltype(g_sgemm)>(p[2]);
    g_out_dim = reinterpret_cast<decltype(g_out_dim)>(p[3]);
    Py_RETURN_NONE;
}

template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
constexpr PyMethodDef method(const char* name) { return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(F)), METH_FASTCALL, nullptr}; }

PyMethodDef g_methods[] = {method<planned>("planned"), method<conv_fwd>("conv_fwd"), method<sgemm>("sgemm"), method<bind>("bind"), {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_torch_calls", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__torch_calls(void) { return PyModule_Create(&g_module); }
