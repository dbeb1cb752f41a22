// The host side of a whole layer's call, as a CPython module.
//
// What bounds a small table's call is the host: marshalled in Python (nine addresses, three allocations through
// the interpreter, two ctypes calls of twenty arguments each) a call of 2 heads of 512 + 128 x 64 kept it busy for
// 22.9 us, where the kernels take 11.7.  Here it is one call with the tensors as they are, 10.7 us on the host, and
// calls follow each other every 16.3 us.  Nothing is computed and nothing is kept: type, sizes, layout and device of
// the arguments are checked, the outputs and the buffer of the codes allocated, and the library's two C entry points,
// whose addresses Python hands in when it loads it, called on the current stream.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "fp8attn.h"

namespace {

decltype(&fp8attn_quantize_qkv_ex) quantize_qkv = nullptr;
decltype(&fp8attn_icl_forward_ex) icl_forward = nullptr;

// bind(address of fp8attn_quantize_qkv_ex, address of fp8attn_icl_forward_ex)
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 2) return PyErr_Format(PyExc_TypeError, "bind takes 2 arguments");
    void* q = PyLong_AsVoidPtr(args[0]);
    void* f = PyLong_AsVoidPtr(args[1]);
    if (PyErr_Occurred()) return nullptr;
    quantize_qkv = reinterpret_cast<decltype(quantize_qkv)>(q);
    icl_forward = reinterpret_cast<decltype(icl_forward)>(f);
    Py_RETURN_NONE;
}

// The tensor of an argument, an undefined one for None; false with an exception set for anything else.
bool tensor(PyObject* o, at::Tensor& t) {
    if (o == Py_None) return true;
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a torch.Tensor");
        return false;
    }
    t = THPVariable_Unpack(o);
    return true;
}

PyObject* refuse(const char* what) {
    PyErr_SetString(PyExc_AssertionError, what);
    return nullptr;
}

// icl_attention(q_train, q_test, k, v, workspace, softmax_scale, flags)
//   -> (status of the quantization, status of the forward call, out_train, out_test)
PyObject* icl_attention(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 7) return PyErr_Format(PyExc_TypeError, "icl_attention takes 7 arguments");
    at::Tensor q_train, q_test, k, v, ws;
    if (!tensor(args[0], q_train) || !tensor(args[1], q_test) || !tensor(args[2], k) || !tensor(args[3], v) ||
        !tensor(args[4], ws))
        return nullptr;
    const double softmax_scale = PyFloat_AsDouble(args[5]);
    const unsigned long flags = PyLong_AsUnsignedLongMask(args[6]);
    if (PyErr_Occurred()) return nullptr;
    if (!k.defined() || k.dim() != 4 || !k.is_cuda() || !k.is_contiguous())
        return refuse("expected contiguous CUDA [B,H,rows,d]");
    if (!q_train.defined() || !v.defined() || !ws.defined()) return refuse("expected tensors");
    const int64_t B = k.size(0), H = k.size(1), n_train = k.size(2), d = k.size(3);
    const int64_t n_test = q_test.defined() ? q_test.size(2) : 0;
    const at::ScalarType type = k.scalar_type();
    if (q_train.scalar_type() != type || v.scalar_type() != type || (n_test > 0 && q_test.scalar_type() != type) ||
        (type != at::kBFloat16 && type != at::kHalf))
        return refuse("expected bf16 or fp16 tensors of one type");
    // The kernels read B * H * rows * d values from each address, as k's sizes have it.
    auto goes_with_k = [&](const at::Tensor& t, int64_t rows) {
        return t.device() == k.device() && t.is_contiguous() && t.dim() >= 2 && t.size(-2) == rows && t.size(-1) == d &&
               t.numel() == B * H * rows * d;
    };
    if (!goes_with_k(q_train, n_train) || !goes_with_k(v, n_train) || (n_test > 0 && !goes_with_k(q_test, n_test)))
        return refuse("expected contiguous tensors of k's batch, heads, d and device");
    if (ws.device() != k.device() || !ws.is_contiguous()) return refuse("expected a contiguous workspace on k's device");
    const bool half = type == at::kHalf, test_only = (flags & FP8ATTN_TEST_ROWS_ONLY) != 0;
    // The codes and scales stay inside this call: one allocation holds them all.
    auto up = [](int64_t x) { return (x + 255) / 256 * 256; };
    const int64_t train = up(B * H * n_train * d), test = up(B * H * n_test * d), scales = up(B * H * 4);
    const at::Tensor codes = at::empty({3 * train + test + 3 * scales}, k.options().dtype(at::kByte));
    at::Tensor out_train, out_test;
    if (!test_only) out_train = at::empty({B, H, n_train, d}, k.options());
    if (n_test > 0) out_test = at::empty({B, H, n_test, d}, k.options());
    char* const q8 = static_cast<char*>(codes.data_ptr());
    char* const k8 = q8 + train;
    char* const v8 = k8 + train;
    char* const t8 = n_test > 0 ? v8 + train : nullptr;
    float* const sq = reinterpret_cast<float*>(v8 + train + test);
    float* const sk = sq + scales / 4;
    float* const sv = sk + scales / 4;
    const void* const x_test = n_test > 0 ? q_test.data_ptr() : nullptr;
    const void* const x_train = q_train.data_ptr();
    const void* const x_k = k.data_ptr();
    const void* const x_v = v.data_ptr();
    void* const o_train = test_only ? nullptr : out_train.data_ptr();
    void* const o_test = n_test > 0 ? out_test.data_ptr() : nullptr;
    void* const w = ws.data_ptr();
    const size_t w_bytes = (size_t)ws.numel();
    void* const stream = c10::cuda::getCurrentCUDAStream().stream();
    int rc_quantize, rc_forward = FP8ATTN_OK;
    Py_BEGIN_ALLOW_THREADS
    rc_quantize = quantize_qkv(x_train, x_k, x_v, x_test, (int)B, (int)H, n_train, n_test, (int)d, q8, k8, v8, t8, sq, sk,
                               sv, half ? FP8ATTN_INPUT_FP16 : 0u, w, w_bytes, stream);
    if (rc_quantize == FP8ATTN_OK)
        rc_forward = icl_forward(test_only ? nullptr : q8, t8, k8, v8, sq, sk, sv, (int)B, (int)H, n_train, n_test, (int)d,
                                 (float)softmax_scale, (uint32_t)flags | (half ? FP8ATTN_IO_FP16 : 0u), o_train, o_test, w,
                                 w_bytes, stream);
    Py_END_ALLOW_THREADS
    PyObject* const a = THPVariable_Wrap(out_train);      // (None for an undefined tensor)
    if (a == nullptr) return nullptr;
    PyObject* const b = THPVariable_Wrap(out_test);
    if (b == nullptr) {
        Py_DECREF(a);
        return nullptr;
    }
    return Py_BuildValue("iiNN", rc_quantize, rc_forward, a, b);
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(bind)), METH_FASTCALL, nullptr},
    {"icl_attention", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(icl_attention)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() { return PyModule_Create(&module); }
