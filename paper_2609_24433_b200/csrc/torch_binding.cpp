// The hot entry points of include/fq.h for torch tensors, as a CPython module: shape and type checks, output and
// workspace from torch's caching allocator, torch's current stream, one call into the library.  Marshalling only, like
// fq.py, which wraps these functions; it is native because an eager call on a short batch is bound by it: the kernels of
// a 64-token projection take 7 us, and a call marshalled through ctypes and torch.empty took 19.4 us of host time
// (at most 8.5 us here, its two launches included; M = 64, K = N = 1024).
//
// Every function returns its result, or the fq_status (an int) of a call that was refused.  All that is read from Python
// objects is read first; then the interpreter lock is given up for the allocations and the call into the library, as ctypes
// and torch do: a launch waits while its stream's queue is full, and other Python threads -- a function that the stream itself
// calls on the host among them, for which that queue may be waiting -- have to run meanwhile.
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

// The interpreter lock given up for a scope, exceptions included.
class Unlocked {
public:
    Unlocked() : state_(PyEval_SaveThread()) {}
    ~Unlocked() { PyEval_RestoreThread(state_); }
    Unlocked(const Unlocked&) = delete;
    Unlocked& operator=(const Unlocked&) = delete;

private:
    PyThreadState* state_;
};

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

// An output: the caller's tensor (its own dtype decides) or, made by make(), a new one of `dtype` on x's device.
struct Output {
    at::Tensor t;
    at::ScalarType type;
    fq_dtype dt;
    Output(PyObject* given, PyObject* dtype) {
        if (!none(given)) {
            t = tensor(given);
            type = t.scalar_type();
        } else if (THPDtype_Check(dtype)) {
            type = reinterpret_cast<THPDtype*>(dtype)->scalar_type;
        } else {
            PyErr_SetString(PyExc_TypeError, "out_dtype has to be a torch.dtype");
            throw Refused();
        }
        dt = dtype_of(type);
    }
    Output(PyObject* given, at::ScalarType otherwise) : type(otherwise), dt(FQ_F32) {
        if (!none(given)) t = tensor(given);
    }
    void make(at::IntArrayRef size, const at::Tensor& like) {
        if (!t.defined()) t = fresh(size, type, like);
    }
};

// The caller's workspace, or one from torch's allocator for the length of the call: it is handed back when the kernels
// are enqueued, and the allocator gives it to later work of this stream only -- what a torch.empty that goes out of
// scope does.
struct Workspace {
    void* p = nullptr;
    size_t bytes = 0;
    at::Tensor own;
    explicit Workspace(PyObject* given) {
        if (none(given)) return;
        const at::Tensor& t = tensor(given);
        p = t.data_ptr();
        bytes = static_cast<size_t>(t.numel());
        given_ = true;
    }
    template <typename Need>
    void make(Need need, const at::Tensor& like) {
        if (given_) return;
        bytes = need();
        own = fresh({static_cast<int64_t>(bytes)}, at::kByte, like);
        p = own.data_ptr();
    }

private:
    bool given_ = false;
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
        const void* xp = x.data_ptr();
        const int64_t ldx = x.stride(0);
        Output y(a[8], a[7]);
        Workspace ws(a[9]);
        fq_status s;
        {
            const Unlocked nogil;
            y.make({M, N}, x);
            ws.make([&] { return fq_workspace_bytes(M, K, N, handle_bits); }, x);
            s = run(which, xp, xt, M, ldx, W, clip, y.t.data_ptr(), y.dt, y.t.stride(0), ws.p, ws.bytes);
        }
        return s == FQ_OK ? THPVariable_Wrap(std::move(y.t)) : status(s);
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
        const void* cp = codes.data_ptr();
        const float* dp = static_cast<const float*>(delta.data_ptr());
        Output y(a[8], a[7]);
        Workspace ws(a[9]);
        fq_status s;
        {
            const Unlocked nogil;
            y.make({M, N}, codes);
            ws.make([&] { return fq_workspace_bytes(M, K, N, handle_bits); }, codes);
            s = (bits == 4 ? fq_gemm_w4a4 : fq_gemm_w8a8)(cp, dp, M, W, y.t.data_ptr(), y.dt, y.t.stride(0), ws.p, ws.bytes, stream());
        }
        return s == FQ_OK ? THPVariable_Wrap(std::move(y.t)) : status(s);
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
        const bool after = integer(a[7]) != 0;
        const void* xp = x.data_ptr();
        const int64_t ldx = x.stride(0);
        Output codes(a[5], at::kByte), delta(a[6], at::kFloat);
        fq_status s;
        {
            const Unlocked nogil;
            codes.make({M, K * bits / 8}, x);
            delta.make({M}, x);
            s = (after ? fq_quantize_act_after : fq_quantize_act)(xp, xt, M, K, ldx, g, block, bits, clip, codes.t.data_ptr(),
                                                                  static_cast<float*>(delta.t.data_ptr()), stream());
        }
        return s == FQ_OK ? pair(std::move(codes.t), std::move(delta.t)) : status(s);
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
        const void* xp = x.data_ptr();
        const int64_t ldx = x.stride(0);
        const int32_t* pp = perm.data_ptr<int32_t>();
        const float* bp = blocks.data_ptr<float>();
        const int block = static_cast<int>(blocks.size(1));
        Output codes(a[6], at::kByte), delta(a[7], at::kFloat);
        Workspace ws(a[8]);
        fq_status s;
        {
            const Unlocked nogil;
            codes.make({M, K * bits / 8}, x);
            delta.make({M}, x);
            ws.make([&] { return static_cast<size_t>(M * K > 4 ? 4 * M * K : 16); }, x);
            s = fq_quantize_act_composite(xp, xt, M, K, ldx, g, pp, bp, block, bits, clip, codes.t.data_ptr(),
                                          static_cast<float*>(delta.t.data_ptr()), ws.p, ws.bytes, stream());
        }
        return s == FQ_OK ? pair(std::move(codes.t), std::move(delta.t)) : status(s);
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
        const void* xp = x.data_ptr();
        const int64_t ldx = x.stride(0);
        Output y(a[4], a[3]);
        fq_status s;
        {
            const Unlocked nogil;
            y.make({M, N}, x);
            s = fq_linear_w4a16(xp, xt, M, ldx, W, y.t.data_ptr(), y.dt, y.t.stride(0), stream());
        }
        return s == FQ_OK ? THPVariable_Wrap(std::move(y.t)) : status(s);
    });
}

#define FQ_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FQ_METHOD(linear), FQ_METHOD(linear_gated), FQ_METHOD(gemm), FQ_METHOD(quantize_act), FQ_METHOD(quantize_act_composite),
                         FQ_METHOD(linear_w4a16), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fq_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fq_torch(void) { return PyModule_Create(&module); }
