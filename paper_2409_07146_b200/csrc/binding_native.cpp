// The decode step's way from torch tensors into libgsa.so, for CPython.  A decode step through a stack of layers is a call
// a layer, each a few microseconds of GPU work: checking seven tensors and marshalling ten arguments in Python took 8.2 us a
// call, more than the kernel.  Here the plain case -- strided CUDA tensors of the expected type and shape, contiguous -- is
// checked and called (24 layers, one sequence, 4 heads of 512: 204 -> 148 us a token, the GPU's pace); anything else is left to
// the Python path (return value None), which words the errors.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "gsa.h"

namespace {

using DecodeStep = gsa_status_t (*)(const gsa_params_t*, const void*, const void*, const void*, const float*, float*, float*, void*,
                                    void*);
DecodeStep g_decode_step = nullptr;

// The address of a plain tensor of this type and shape; null for anything else (subclasses, wrappers without storage, other
// layouts, devices, types, shapes and strides).
void* plain(PyObject* obj, at::ScalarType type, std::initializer_list<int64_t> shape) {
    if (!THPVariable_CheckExact(obj)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(obj);
    if (!t.defined() || !t.has_storage() || t.layout() != at::kStrided || !t.is_cuda() || t.scalar_type() != type) return nullptr;
    if (!t.is_contiguous() || t.sizes() != at::IntArrayRef(shape.begin(), shape.size())) return nullptr;
    return t.data_ptr();
}

// decode_step(params address, q, k, v, gate, K, V, o) -> status, or None: not a plain call
PyObject* decode_step(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 8 || g_decode_step == nullptr) Py_RETURN_NONE;
    const void* at = PyLong_AsVoidPtr(args[0]);
    if (at == nullptr) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    const gsa_params_t& p = *static_cast<const gsa_params_t*>(at);
    const at::ScalarType io = p.io == GSA_BF16 ? at::kBFloat16 : at::kFloat, gt = p.gate_dtype == GSA_BF16 ? at::kBFloat16 : at::kFloat;
    try {
        const void* q = plain(args[1], io, {p.B, p.H, p.d_k});
        const void* k = plain(args[2], io, {p.B, p.H, p.d_k});
        const void* v = plain(args[3], io, {p.B, p.H, p.d_v});
        const void* gate = p.gate_broadcast ? plain(args[4], gt, {p.H, p.m}) : plain(args[4], gt, {p.B, p.H, p.m});
        void* K = plain(args[5], at::kFloat, {p.B, p.H, p.m, p.d_k});
        void* V = plain(args[6], at::kFloat, {p.B, p.H, p.m, p.d_v});
        void* o = plain(args[7], io, {p.B, p.H, p.d_v});
        if (!q || !k || !v || !gate || !K || !V || !o) Py_RETURN_NONE;
        void* stream = c10::cuda::getCurrentCUDAStream().stream();
        gsa_status_t rc;
        Py_BEGIN_ALLOW_THREADS
        rc = g_decode_step(&p, q, k, v, static_cast<const float*>(gate), static_cast<float*>(K), static_cast<float*>(V), o, stream);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong((long)rc);
    } catch (...) {             // (torch's exceptions: the Python path meets them again and reports them)
        Py_RETURN_NONE;
    }
}

// set_library(address of gsa_decode_step)
PyObject* set_library(PyObject*, PyObject* address) {
    void* at = PyLong_AsVoidPtr(address);
    if (at == nullptr && PyErr_Occurred()) return nullptr;
    g_decode_step = reinterpret_cast<DecodeStep>(at);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"decode_step", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(decode_step)), METH_FASTCALL, nullptr},
    {"set_library", set_library, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
