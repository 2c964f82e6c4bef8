// The hot entry points of include/fq.h for torch tensors, as a CPython module: shape and type checks, output and
// workspace from torch's caching allocator, torch's current stream, one call into the library.  Marshalling only, like
// fq.py, which wraps these functions; it is native because an eager call on a short batch is bound by it: the kernels of
// a 64-token projection take 7 us, and a call marshalled through ctypes and torch.empty took 19.4 us of host time
// (at most 8.5 us here, its two launches included; M = 64, K = N = 1024).
//
// Every function returns its result, or the fq_status (an int) of a call that was refused.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "fq.h"

namespace {

struct Refused {};          // a Python exception is set

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "expected a torch.Tensor, got %s", Py_TYPE(o)->tp_name);
        throw Refused();
    }
    return THPVariable_Unpack(o);
}
const at::Tensor& rowmajor(PyObject* o) {
    const at::Tensor& t = tensor(o);
    if (t.dim() != 2 || t.stride(1) != 1) {
        PyErr_SetString(PyExc_ValueError, "expected a 2-D tensor with unit inner stride");
        throw Refused();
    }
    return t;
}
long long integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Refused();
    return v;
}
void* address(PyObject* o) { return reinterpret_cast<void*>(static_cast<uintptr_t>(integer(o))); }
float real(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Refused();
    return static_cast<float>(v);
}
fq_dtype dtype_of(at::ScalarType t) {
    if (t == at::kFloat) return FQ_F32;
    if (t == at::kBFloat16) return FQ_BF16;
    PyErr_Format(PyExc_TypeError, "unsupported dtype %s", at::toString(t));
    throw Refused();
}
void arguments(Py_ssize_t got, Py_ssize_t wanted) {
    if (got != wanted) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", wanted, got);
        throw Refused();
    }
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
bool none(PyObject* o) { return o == Py_None; }
PyObject* status(fq_status s) { return PyLong_FromLong(s); }

// (on a GPU straight from the allocator: at::empty's way through the dispatcher costs as much again)
at::Tensor fresh(at::IntArrayRef size, at::ScalarType t, const at::Tensor& like) {
    if (like.is_cuda()) return at::Tensor(at::detail::empty_cuda(size, t, like.device(), std::nullopt));
    return at::empty(size, at::TensorOptions().dtype(t).device(like.device()));
}

// y as given (its own dtype decides) or a new [M, N] of `dtype` on x's device
at::Tensor output(PyObject* y, PyObject* dtype, int64_t M, int64_t N, const at::Tensor& x, fq_dtype* yt) {
    if (!none(y)) {
        const at::Tensor& t = tensor(y);
        *yt = dtype_of(t.scalar_type());
        return t;
    }
    if (!THPDtype_Check(dtype)) {
        PyErr_SetString(PyExc_TypeError, "out_dtype has to be a torch.dtype");
        throw Refused();
    }
    const at::ScalarType t = reinterpret_cast<THPDtype*>(dtype)->scalar_type;
    *yt = dtype_of(t);
    return fresh({M, N}, t, x);
}

// The caller's workspace, or one from torch's allocator for the length of the call: it is handed back when the kernels
// are enqueued, and the allocator gives it to later work of this stream only -- what a torch.empty that goes out of
// scope does.
struct Workspace {
    void* p = nullptr;
    size_t bytes = 0;
    at::Tensor own;
    Workspace(PyObject* given, size_t need, const at::Tensor& like) {
        if (!none(given)) {
            const at::Tensor& t = tensor(given);
            p = t.data_ptr();
            bytes = static_cast<size_t>(t.numel());
        } else {
            own = fresh({static_cast<int64_t>(need)}, at::kByte, like);
            p = own.data_ptr();
            bytes = need;
        }
    }
};

PyObject* pair(at::Tensor&& a, at::Tensor&& b) {
    PyObject* r = PyTuple_New(2);
    if (!r) return nullptr;
    PyTuple_SET_ITEM(r, 0, THPVariable_Wrap(std::move(a)));
    PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(std::move(b)));
    return r;
}

template <typename F>
PyObject* guarded(F f) {
    HANDLE_TH_ERRORS
    try {
        return f();
    } catch (const Refused&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// The arguments that the one-call entry points share: (x, handle, K, N, handle_bits, ., clip_ratio, out_dtype, y, workspace)
template <typename F>
PyObject* one_call(PyObject* const* a, Py_ssize_t n, F run) {
    return guarded([&]() -> PyObject* {
        arguments(n, 10);
        const at::Tensor& x = rowmajor(a[0]);
        const fq_weights* W = static_cast<const fq_weights*>(address(a[1]));
        const int64_t K = integer(a[2]), N = integer(a[3]), M = x.size(0);
        const int handle_bits = static_cast<int>(integer(a[4]));
        const long long which = integer(a[5]);
        const float clip = real(a[6]);
        const fq_dtype xt = dtype_of(x.scalar_type());
        fq_dtype yt;
        at::Tensor y = output(a[8], a[7], M, N, x, &yt);
        const Workspace ws(a[9], none(a[9]) ? fq_workspace_bytes(M, K, N, handle_bits) : 0, x);
        const fq_status s = run(which, x.data_ptr(), xt, M, x.stride(0), W, clip, y.data_ptr(), yt, y.stride(0), ws.p, ws.bytes);
        return s == FQ_OK ? THPVariable_Wrap(std::move(y)) : status(s);
    });
}

// linear(x, handle, K, N, handle_bits, bits, clip_ratio, out_dtype, y, workspace): fq_linear_w4a4 / _w8a8 by `bits`
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return one_call(a, n, [](long long bits, const void* x, fq_dtype xt, int64_t M, int64_t ldx, const fq_weights* W, float clip,
                             void* y, fq_dtype yt, int64_t ldy, void* ws, size_t ws_bytes) {
        return (bits == 4 ? fq_linear_w4a4 : fq_linear_w8a8)(x, xt, M, ldx, W, clip, y, yt, ldy, ws, ws_bytes, stream());
    });
}

// linear_gated(x, handle, K, N, handle_bits, act, clip_ratio, out_dtype, y, workspace): fq_linear_gated.  (`act` is the
// caller's: whatever is neither function is refused as the library refuses it, ahead of its narrowing to the enumeration.)
PyObject* linear_gated(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return one_call(a, n, [](long long act, const void* x, fq_dtype xt, int64_t M, int64_t ldx, const fq_weights* W, float clip,
                             void* y, fq_dtype yt, int64_t ldy, void* ws, size_t ws_bytes) {
        if (act != FQ_GATE_SILU && act != FQ_GATE_GELU_TANH) return FQ_ERR_INVALID_ARG;
        return fq_linear_gated(x, xt, M, ldx, static_cast<fq_gate_act>(act), W, clip, y, yt, ldy, ws, ws_bytes, stream());
    });
}

// gemm(codes, delta, handle, K, N, handle_bits, bits, out_dtype, y, workspace): fq_gemm_w4a4 / fq_gemm_w8a8 by `bits`
PyObject* gemm(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        arguments(n, 10);
        const at::Tensor &codes = tensor(a[0]), &delta = tensor(a[1]);
        const fq_weights* W = static_cast<const fq_weights*>(address(a[2]));
        const int64_t K = integer(a[3]), N = integer(a[4]), M = codes.size(0);
        const int handle_bits = static_cast<int>(integer(a[5])), bits = static_cast<int>(integer(a[6]));
        fq_dtype yt;
        at::Tensor y = output(a[8], a[7], M, N, codes, &yt);
        const Workspace ws(a[9], none(a[9]) ? fq_workspace_bytes(M, K, N, handle_bits) : 0, codes);
        const fq_status s = (bits == 4 ? fq_gemm_w4a4 : fq_gemm_w8a8)(codes.data_ptr(), static_cast<const float*>(delta.data_ptr()), M,
                                                                      W, y.data_ptr(), yt, y.stride(0), ws.p, ws.bytes, stream());
        return s == FQ_OK ? THPVariable_Wrap(std::move(y)) : status(s);
    });
}

// quantize_act(x, multiplier address, block, bits, clip_ratio, codes, delta, fold_after) -> (codes, delta)
PyObject* quantize_act(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        arguments(n, 8);
        const at::Tensor& x = rowmajor(a[0]);
        const float* g = static_cast<const float*>(address(a[1]));
        const int64_t M = x.size(0), K = x.size(1);
        const int block = static_cast<int>(integer(a[2])), bits = static_cast<int>(integer(a[3]));
        const float clip = real(a[4]);
        const fq_dtype xt = dtype_of(x.scalar_type());
        at::Tensor codes = none(a[5]) ? fresh({M, K * bits / 8}, at::kByte, x) : tensor(a[5]);
        at::Tensor delta = none(a[6]) ? fresh({M}, at::kFloat, x) : tensor(a[6]);
        const fq_status s = (integer(a[7]) ? fq_quantize_act_after : fq_quantize_act)(
            x.data_ptr(), xt, M, K, x.stride(0), g, block, bits, clip, codes.data_ptr(), static_cast<float*>(delta.data_ptr()), stream());
        return s == FQ_OK ? pair(std::move(codes), std::move(delta)) : status(s);
    });
}

// quantize_act_composite(x, multiplier address, perm, blocks, bits, clip_ratio, codes, delta, workspace) -> (codes, delta)
PyObject* quantize_act_composite(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        arguments(n, 9);
        const at::Tensor& x = rowmajor(a[0]);
        const float* g = static_cast<const float*>(address(a[1]));
        const at::Tensor &perm = tensor(a[2]), &blocks = tensor(a[3]);
        if (perm.scalar_type() != at::kInt || blocks.scalar_type() != at::kFloat || !blocks.is_contiguous() || blocks.dim() != 3) {
            PyErr_SetString(PyExc_AssertionError, "perm has to be int32, blocks contiguous float32 [K/block, block, block]");
            throw Refused();
        }
        const int64_t M = x.size(0), K = x.size(1);
        const int bits = static_cast<int>(integer(a[4]));
        const float clip = real(a[5]);
        const fq_dtype xt = dtype_of(x.scalar_type());
        at::Tensor codes = none(a[6]) ? fresh({M, K * bits / 8}, at::kByte, x) : tensor(a[6]);
        at::Tensor delta = none(a[7]) ? fresh({M}, at::kFloat, x) : tensor(a[7]);
        const Workspace ws(a[8], static_cast<size_t>(M * K > 4 ? 4 * M * K : 16), x);
        const fq_status s = fq_quantize_act_composite(x.data_ptr(), xt, M, K, x.stride(0), g, perm.data_ptr<int32_t>(),
                                                      blocks.data_ptr<float>(), static_cast<int>(blocks.size(1)), bits, clip,
                                                      codes.data_ptr(), static_cast<float*>(delta.data_ptr()), ws.p, ws.bytes, stream());
        return s == FQ_OK ? pair(std::move(codes), std::move(delta)) : status(s);
    });
}

// linear_w4a16(x, handle, N, out_dtype, y)
PyObject* linear_w4a16(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        arguments(n, 5);
        const at::Tensor& x = rowmajor(a[0]);
        const fq_weights* W = static_cast<const fq_weights*>(address(a[1]));
        const int64_t N = integer(a[2]), M = x.size(0);
        const fq_dtype xt = dtype_of(x.scalar_type());
        fq_dtype yt;
        at::Tensor y = output(a[4], a[3], M, N, x, &yt);
        const fq_status s = fq_linear_w4a16(x.data_ptr(), xt, M, x.stride(0), W, y.data_ptr(), yt, y.stride(0), stream());
        return s == FQ_OK ? THPVariable_Wrap(std::move(y)) : status(s);
    });
}

#define FQ_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FQ_METHOD(linear), FQ_METHOD(linear_gated), FQ_METHOD(gemm), FQ_METHOD(quantize_act), FQ_METHOD(quantize_act_composite),
                         FQ_METHOD(linear_w4a16), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fq_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fq_torch(void) { return PyModule_Create(&module); }
