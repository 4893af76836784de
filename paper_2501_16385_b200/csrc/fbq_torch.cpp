// Native marshalling of torch tensors into the C ABI of libfbq.so (module _fbq_torch): the part of the Python binding
// that a decode loop runs once per linear.  A linear at one token takes the GPU about five microseconds; marshalling
// its fourteen arguments in Python and through ctypes took the host more than ten (4096 -> 4096, INT4, rank 32, call
// after call: 15.2 us per call before, 4.2 us to issue and 5.7 us in all now).
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>

#include "../../include/fbq.h"

namespace {

// A tensor argument's address (NULL for None); false with an exception set when it is neither.
bool address(PyObject *o, void **out)
{
    if (o == Py_None) {
        *out = nullptr;
        return true;
    }
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a tensor");
        return false;
    }
    *out = THPVariable_Unpack(o).data_ptr();
    return true;
}

bool stream_of(PyObject *o, void **out)
{
    if (o == Py_None) {
        *out = static_cast<void *>(c10::cuda::getCurrentCUDAStream().stream());
        return true;
    }
    PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) return false;
    *out = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
}

// linear(x, qweight, scales, zeros, A, B, N, group, bits, y, stream) -> y, or the error code of the call
PyObject *py_linear(PyObject *, PyObject *const *v, Py_ssize_t n)
{
    if (n != 11) {
        PyErr_SetString(PyExc_TypeError, "linear takes 11 arguments");
        return nullptr;
    }
    try {
        if (!THPVariable_Check(v[0])) {
            PyErr_SetString(PyExc_TypeError, "expected a tensor");
            return nullptr;
        }
        const at::Tensor &x = THPVariable_Unpack(v[0]);
        if (!x.is_cuda() || !x.is_contiguous() || x.dim() != 2) {
            PyErr_SetString(PyExc_AssertionError, "x must be a contiguous CUDA matrix");
            return nullptr;
        }
        const bool f16 = x.scalar_type() == at::kHalf;
        if (!f16 && x.scalar_type() != at::kBFloat16) {
            PyErr_SetString(PyExc_TypeError, "x must be float16 or bfloat16");
            return nullptr;
        }
        const int64_t M = x.size(0), K = x.size(1);
        const long N = PyLong_AsLong(v[6]), group = PyLong_AsLong(v[7]), bits = PyLong_AsLong(v[8]);
        if (PyErr_Occurred()) return nullptr;
        int64_t rank = 0;
        if (v[4] != Py_None) {
            if (!THPVariable_Check(v[4])) {
                PyErr_SetString(PyExc_TypeError, "expected a tensor");
                return nullptr;
            }
            rank = THPVariable_Unpack(v[4]).size(0);
        }
        void *p[6], *stream;
        for (int i = 1; i < 6; ++i)
            if (!address(v[i], &p[i])) return nullptr;
        if (!stream_of(v[10], &stream)) return nullptr;
        PyObject *y;
        if (v[9] == Py_None) {
            y = THPVariable_Wrap(at::empty({M, (int64_t)N}, x.options()));
            if (!y) return nullptr;
        } else {
            y = v[9];
            Py_INCREF(y);
        }
        void *yp;
        if (!address(y, &yp)) {
            Py_DECREF(y);
            return nullptr;
        }
        void *xp = x.data_ptr();
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = (f16 ? fbq_linear : fbq_linear_bf16)(xp, static_cast<const uint32_t *>(p[1]), p[2], p[3], p[4], p[5], yp, (int)M, (int)N, (int)K,
                                                  (int)group, (int)bits, (int)rank, stream);
        Py_END_ALLOW_THREADS
        if (rc == FBQ_OK) return y;
        Py_DECREF(y);
        return PyLong_FromLong(rc);
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// linear_batch(address of the descriptors, count, M, group, bits, rank, bf16, host_io, stream) -> error code
PyObject *py_linear_batch(PyObject *, PyObject *const *v, Py_ssize_t n)
{
    if (n != 9) {
        PyErr_SetString(PyExc_TypeError, "linear_batch takes 9 arguments");
        return nullptr;
    }
    const fbq_problem *problems = static_cast<const fbq_problem *>(PyLong_AsVoidPtr(v[0]));
    int a[7];
    for (int i = 0; i < 7; ++i) a[i] = (int)PyLong_AsLong(v[i + 1]);
    if (PyErr_Occurred()) return nullptr;
    void *stream;
    if (!stream_of(v[8], &stream)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = (a[6] ? fbq_linear_batch_hostio : fbq_linear_batch)(problems, a[0], a[1], a[2], a[3], a[4], a[5], stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

PyMethodDef methods[] = {{"linear", (PyCFunction)(void (*)(void))py_linear, METH_FASTCALL, nullptr},
                         {"linear_batch", (PyCFunction)(void (*)(void))py_linear_batch, METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fbq_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fbq_torch() { return PyModule_Create(&module); }
