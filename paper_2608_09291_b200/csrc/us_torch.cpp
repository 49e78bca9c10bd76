// The per-call half of the Python front end (binding.py): takes the caller's torch tensors apart, makes the
// output, finds the stream and calls the C ABI, in native code. Torch tensors are used only as device memory.
//
// A decode-sized product takes 3 to 5 us on the GPU. Marshalling the call in Python took 9.3 us (an output tensor
// 2.5, the current stream 2.2, ctypes with the launch 3.1, the rest argument handling), so every product up to
// about 8 us of GPU time was bound by it; the calls below leave 0.6 us around the launch's own 1.8.
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>

#include "../../include/unionsparse.h"

namespace {

PyObject* g_error = nullptr;   // binding.UsError

PyObject* fail(us_status s, const char* where)
{
    if (!g_error) return PyErr_Format(PyExc_RuntimeError, "%s: status %d", where, (int)s);
    PyObject* e = PyObject_CallFunction(g_error, "is", (int)s, where);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    return nullptr;
}

// A tensor argument; nullptr with an error set if it is none.
const at::Tensor* tensor(PyObject* o, const char* name)
{
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a torch.Tensor, not %s", name, Py_TYPE(o)->tp_name);
        return nullptr;
    }
    return &THPVariable_Unpack(o);
}

// Optional tensor argument: None gives a null pointer.
bool pointer(PyObject* o, const char* name, void** out)
{
    *out = nullptr;
    if (o == Py_None) return true;
    const at::Tensor* t = tensor(o, name);
    if (!t) return false;
    *out = t->data_ptr();
    return true;
}

bool stream_of(PyObject* o, const at::Tensor& on, void** out)
{
    if (o != Py_None) {
        *out = PyLong_AsVoidPtr(o);
        return !PyErr_Occurred();
    }
    if (!on.is_cuda()) {
        PyErr_SetString(PyExc_ValueError, "expected a tensor on a CUDA device");
        return false;
    }
    *out = c10::cuda::getCurrentCUDAStream(on.device().index()).stream();
    return true;
}

bool is_f16_rows(const at::Tensor& t) { return t.scalar_type() == at::kHalf && t.dim() == 2 && t.stride(1) == 1; }

// The caller's output tensor, or a new one on the device of `on`.
at::Tensor new_output(const at::Tensor& on, int64_t N, int64_t M, at::ScalarType type)
{
    const int64_t shape[2] = {N, M};
    if (on.is_cuda()) return at::detail::empty_cuda(shape, type, on.device(), std::nullopt);
    return at::empty(shape, on.options().dtype(type));
}

// spmm(handle, M, X, N, x_scale, out, stream) -> the output tensor
PyObject* spmm(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 7) return PyErr_Format(PyExc_TypeError, "spmm takes 7 arguments");
    HANDLE_TH_ERRORS
    void *h = nullptr, *xs = nullptr, *st = nullptr;
    if (a[0] != Py_None) h = PyLong_AsVoidPtr(a[0]);
    const int64_t M = PyLong_AsLongLong(a[1]);
    const int64_t N = PyLong_AsLongLong(a[3]);
    if (PyErr_Occurred()) return nullptr;
    const at::Tensor* X = tensor(a[2], "X");
    if (!X || !pointer(a[4], "x_scale", &xs) || !stream_of(a[6], *X, &st)) return nullptr;
    if (N < 1 || N > 64) return fail(US_ERR_INVALID_ARG, "us_spmm");
    at::Tensor fresh;
    const at::Tensor* out = nullptr;
    if (a[5] != Py_None) {
        out = tensor(a[5], "out");
        if (!out) return nullptr;
    } else {
        fresh = new_output(*X, N, M, xs ? at::kHalf : at::kInt);
    }
    us_status s;
    void* y = out ? out->data_ptr() : fresh.data_ptr();
    Py_BEGIN_ALLOW_THREADS
    s = us_spmm(static_cast<us_handle*>(h), X->data_ptr(), (int32_t)N, xs, y, st);
    Py_END_ALLOW_THREADS
    if (s != US_OK) return fail(s, "us_spmm");
    if (out) {
        Py_INCREF(a[5]);
        return a[5];
    }
    return THPVariable_Wrap(std::move(fresh));
    END_HANDLE_TH_ERRORS
}

// spmm_requant(handle, M, K, X16, N, x_amax, out, y_amax, m0, m1, stream) -> the output tensor
PyObject* spmm_requant(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 11) return PyErr_Format(PyExc_TypeError, "spmm_requant takes 11 arguments");
    HANDLE_TH_ERRORS
    void *h = nullptr, *xa = nullptr, *ya = nullptr, *st = nullptr;
    if (a[0] != Py_None) h = PyLong_AsVoidPtr(a[0]);
    const int64_t M = PyLong_AsLongLong(a[1]), K = PyLong_AsLongLong(a[2]), N = PyLong_AsLongLong(a[4]);
    const int64_t m0 = PyLong_AsLongLong(a[8]), m1 = PyLong_AsLongLong(a[9]);
    if (PyErr_Occurred()) return nullptr;
    const at::Tensor* X = tensor(a[3], "X16");
    if (!X || !pointer(a[5], "x_amax", &xa) || !pointer(a[7], "y_amax", &ya) || !stream_of(a[10], *X, &st)) return nullptr;
    if (!is_f16_rows(*X) || X->size(1) != K)
        return PyErr_Format(PyExc_AssertionError, "X16 must be a float16 (N, K) tensor with unit column stride");
    if (N < 1 || N > 64) return fail(US_ERR_INVALID_ARG, "us_spmm_requant");
    at::Tensor fresh;
    const at::Tensor* out = nullptr;
    if (a[6] != Py_None) {
        out = tensor(a[6], "out");
        if (!out) return nullptr;
    } else {
        fresh = new_output(*X, N, M, at::kHalf);
    }
    us_status s;
    void* y = out ? out->data_ptr() : fresh.data_ptr();
    const int64_t ldx = X->stride(0);
    Py_BEGIN_ALLOW_THREADS
    s = us_spmm_requant(static_cast<us_handle*>(h), X->data_ptr(), ldx, xa, (int32_t)N, y, ya, m0, m1, st);
    Py_END_ALLOW_THREADS
    if (s != US_OK) return fail(s, "us_spmm_requant");
    if (out) {
        Py_INCREF(a[6]);
        return a[6];
    }
    return THPVariable_Wrap(std::move(fresh));
    END_HANDLE_TH_ERRORS
}

// absmax_f16(X16, amax, stream)
PyObject* absmax_f16(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (n != 3) return PyErr_Format(PyExc_TypeError, "absmax_f16 takes 3 arguments");
    HANDLE_TH_ERRORS
    void *am = nullptr, *st = nullptr;
    const at::Tensor* X = tensor(a[0], "X16");
    if (!X || !pointer(a[1], "amax", &am) || !stream_of(a[2], *X, &st)) return nullptr;
    if (!is_f16_rows(*X)) return PyErr_Format(PyExc_AssertionError, "X16 must be a float16 (N, K) tensor with unit column stride");
    const int64_t N = X->size(0);
    if (N < 1 || N > 64) return fail(US_ERR_INVALID_ARG, "us_absmax_f16");
    us_status s;
    Py_BEGIN_ALLOW_THREADS
    s = us_absmax_f16(X->data_ptr(), X->stride(0), (int32_t)N, X->size(1), am, st);
    Py_END_ALLOW_THREADS
    if (s != US_OK) return fail(s, "us_absmax_f16");
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

PyObject* set_error(PyObject*, PyObject* cls)
{
    Py_XDECREF(g_error);
    Py_INCREF(cls);
    g_error = cls;
    Py_RETURN_NONE;
}

template <class F>
PyCFunction fast(F* f) { return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)); }

PyMethodDef methods[] = {
    {"spmm", fast(spmm), METH_FASTCALL, nullptr},
    {"spmm_requant", fast(spmm_requant), METH_FASTCALL, nullptr},
    {"absmax_f16", fast(absmax_f16), METH_FASTCALL, nullptr},
    {"set_error", set_error, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_us_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__us_torch() { return PyModule_Create(&module); }
