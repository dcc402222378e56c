// CPython entry of the product for calls whose buffers the caller holds (out and workspace given, current stream): the
// same checks and the same C ABI call as binding.gemm, without its ~8 us of Python per call (attribute look-ups, shape
// tuples, ctypes conversions), which is what bounded the small products (1 x 16 x 512 x 512: 12.5 us a call, 7.1 now; 1 x 1 x 4096 x 4096: 15.3 and 11.0).
// Anything it does not take as it is (another type, shape, layout or device, a tensor subclass or wrapper) returns
// None: the caller then goes through binding.gemm's own checks and gets their error, or their call.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>

namespace {

typedef int (*GemmExFn)(const void*, const void*, const uint32_t*, const float*, const void*, void*, int, int, int, int, int,
                        int, void*, size_t, void*);
GemmExFn g_gemm_ex = nullptr;   // of the library the binding has loaded

// Address of the library's bitdelta_gemm_ex (as an integer).
PyObject* set_library(PyObject*, PyObject* arg) {
    void* p = PyLong_AsVoidPtr(arg);
    if (PyErr_Occurred()) return nullptr;
    g_gemm_ex = reinterpret_cast<GemmExFn>(p);
    Py_RETURN_NONE;
}

// A plain torch.Tensor (no subclass) on a CUDA device, contiguous, of `type`.
bool plain(PyObject* o, c10::ScalarType type) {
    if (!THPVariable_CheckExact(o)) return false;
    const at::Tensor& t = THPVariable_Unpack(o);
    return t.is_cuda() && t.scalar_type() == type && t.is_contiguous();
}

// (X, W_base, bits, alpha, bias or None, out, workspace, dtype flags beyond the element type, activation code) ->
// status of the call, or None.
PyObject* gemm(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 9 || !g_gemm_ex) Py_RETURN_NONE;
    try {
        if (!THPVariable_CheckExact(a[0])) Py_RETURN_NONE;
        const at::Tensor& X = THPVariable_Unpack(a[0]);
        const c10::ScalarType io = X.scalar_type();
        if (io != c10::ScalarType::BFloat16 && io != c10::ScalarType::Half) Py_RETURN_NONE;
        const bool has_bias = a[4] != Py_None;
        if (!plain(a[0], io) || !plain(a[1], io) || !plain(a[2], c10::ScalarType::Int) || !plain(a[3], c10::ScalarType::Float) ||
            (has_bias && !plain(a[4], io)) || !plain(a[5], io) || !THPVariable_CheckExact(a[6]))
            Py_RETURN_NONE;
        const at::Tensor &W = THPVariable_Unpack(a[1]), &bits = THPVariable_Unpack(a[2]), &alpha = THPVariable_Unpack(a[3]);
        const at::Tensor &out = THPVariable_Unpack(a[5]), &ws = THPVariable_Unpack(a[6]);
        if (X.dim() != 3 || W.dim() != 2 || bits.dim() != 3 || alpha.dim() != 1) Py_RETURN_NONE;
        const int64_t B = X.size(0), m = X.size(1), K = X.size(2), N = W.size(0);
        if (W.size(1) != K || bits.size(0) != B || bits.size(1) != N || bits.size(2) != K / 32 || alpha.size(0) != B)
            Py_RETURN_NONE;
        if (B > INT32_MAX || m > INT32_MAX || K > INT32_MAX || N > INT32_MAX) Py_RETURN_NONE;
        const void* bias = nullptr;
        if (has_bias) {
            const at::Tensor& b = THPVariable_Unpack(a[4]);
            if (b.dim() != 1 || b.size(0) != N) Py_RETURN_NONE;
            bias = b.data_ptr();
        }
        const long flags = PyLong_AsLong(a[7]), act = PyLong_AsLong(a[8]);
        if (PyErr_Occurred()) return nullptr;
        if (act == 2 && (N % 2) != 0) Py_RETURN_NONE;
        const void *px = X.data_ptr(), *pw = W.data_ptr(), *pb = bits.data_ptr(), *pa = alpha.data_ptr();
        void *po = out.data_ptr(), *pws = ws.data_ptr();
        const size_t ws_bytes = (size_t)ws.numel();
        void* stream = c10::cuda::getCurrentCUDAStream().stream();
        int st;
        Py_BEGIN_ALLOW_THREADS
        st = g_gemm_ex(px, pw, static_cast<const uint32_t*>(pb), static_cast<const float*>(pa), bias, po, (int)B, (int)m, (int)N,
                       (int)K, (int)flags | (io == c10::ScalarType::Half ? 1 : 0), (int)act, pws, ws_bytes, stream);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(st);
    } catch (...) {   // (a wrapped tensor without storage, for one: binding.gemm raises what it always has)
        if (PyErr_Occurred()) PyErr_Clear();
        Py_RETURN_NONE;
    }
}

PyMethodDef methods[] = {
    {"set_library", set_library, METH_O, "Address of bitdelta_gemm_ex in the loaded library."},
    {"gemm", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(gemm)), METH_FASTCALL, "The product; None if the call is not a plain one."},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall(void) { return PyModule_Create(&module); }
