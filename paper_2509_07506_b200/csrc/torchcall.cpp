// Direct calls of the astra.h ABI on torch tensors, without Python-level checks: the second half of the
// _astra_fastcall extension.
//
// A direct call from the binding's Python code costs 3.5 to 12 us of attribute reads, checks and argument
// conversions, more than the launch and far more than the kernel of a decode-sized shape.  Each function
// here makes the same checks on the tensors' C++ objects and hands addresses and the current stream to the
// entry point.  It answers the ordinary case only: whenever a check does not hold, or anything about an
// operand is unusual (a tensor subclass, a functorch or functionalisation wrapper, an active torch-function
// mode, another current device), it returns None without having launched anything, and the binding takes
// its own route, which launches or raises the precise error.  Otherwise it returns the entry point's status;
// every argument check of the C ABI still runs there.
// Host time per call, enqueued back to back, Python-level checks -> here (a prepared call: 2.2 us, nearly all
// of it the launch): rmsnorm 5.1 -> 2.3 us, silu 5.0 -> 2.5, merge 7.4 -> 2.6, all-reduce with 8 partials 11.7 ->
// 2.9; the strided forms, which went through ctypes, 12.8 -> 2.2, 10.3 -> 2.5, 15.1 -> 2.7, and 26.6 -> 3.4 us
// with 8 partials and 8 destinations.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/core/TensorBase.h>
#include <c10/core/DispatchKeySet.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/version.h>

#include <algorithm>
#include <exception>
#include <type_traits>

#include "astra.h"
#include "fastcall.h"

namespace {

constexpr int kMaxTable = 16;

// Returned for "not the ordinary case".
struct Unusual {};

const at::TensorBase &tensor(PyObject *o) {
    if (!THPVariable_CheckExact(o)) throw Unusual();  // Tensor or Parameter, no subclass
    const at::TensorBase &t = THPVariable_Unpack(o);
    static const c10::DispatchKeySet wrappers({c10::DispatchKey::Python, c10::DispatchKey::Functionalize,
                                               c10::DispatchKey::FuncTorchBatched, c10::DispatchKey::FuncTorchGradWrapper,
                                               c10::DispatchKey::Batched, c10::DispatchKey::Negative,
                                               c10::DispatchKey::Conjugate, c10::DispatchKey::ZeroTensor});
    if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || !t.has_storage() || t.key_set().has_any(wrappers))
        throw Unusual();
    return t;
}

astra_dtype_t dtype_of(const at::TensorBase &t) {
    switch (t.scalar_type()) {
        case at::kBFloat16: return ASTRA_BF16;
        case at::kHalf: return ASTRA_FP16;
        case at::kFloat: return ASTRA_FP32;
        default: throw Unusual();
    }
}

inline void require(bool ok) {
    if (!ok) throw Unusual();
}

// Same dtype and shape as `like`, contiguous, on its device (unless it may be a peer's).
void *dense(PyObject *o, const at::TensorBase &like, at::IntArrayRef sizes, bool any_device = false) {
    const at::TensorBase &t = tensor(o);
    require(t.scalar_type() == like.scalar_type() && t.sizes() == sizes && t.is_contiguous() &&
            (any_device || t.device() == like.device()));
    return t.mutable_data_ptr();
}

void *scores(PyObject *o, const at::TensorBase &like, at::IntArrayRef sizes) {
    const at::TensorBase &t = tensor(o);
    require(t.scalar_type() == at::kFloat && t.sizes() == sizes && t.is_contiguous() && t.device() == like.device());
    return t.mutable_data_ptr();
}

// Same dtype, shape and device as `like`, innermost dimension contiguous.
const at::TensorBase &rows(PyObject *o, const at::TensorBase &like) {
    const at::TensorBase &t = tensor(o);
    require(t.scalar_type() == like.scalar_type() && t.sizes() == like.sizes() && t.device() == like.device() &&
            (t.size(-1) <= 1 || t.stride(-1) == 1));
    return t;
}

// A single row may report any stride; its width is used then.
int64_t pitch(const at::TensorBase &t) {
    return t.size(0) > 1 ? t.stride(0) : std::max<int64_t>(t.stride(0), t.size(1));
}

float number(PyObject *o) {
    require(PyFloat_Check(o) || PyLong_CheckExact(o));
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Unusual();
    return static_cast<float>(v);
}

// The stream to launch on; the call's device must be current, since the C side launches on that one.
void *stream_of(PyObject *stream, const at::TensorBase &t) {
    require(!at::impl::torch_function_mode_enabled());
    const c10::DeviceIndex dev = t.device().index();
    require(dev == c10::cuda::current_device());
    if (stream == Py_None) return c10::cuda::getCurrentCUDAStream(dev).stream();
    PyObject *handle = PyObject_GetAttrString(stream, "cuda_stream");
    require(handle != nullptr);
    void *p = PyLong_Check(handle) ? PyLong_AsVoidPtr(handle) : nullptr;
    const bool known = PyLong_Check(handle) && !PyErr_Occurred();
    Py_DECREF(handle);
    require(known);
    return p;
}

// Addresses of 1 to 16 dense tensors in a list or tuple; they may live on other GPUs.
// The table holds references: a list may be changed by another thread while the call runs unlocked.
struct Table {
    void *p[kMaxTable];
    PyObject *held[kMaxTable];
    int n = 0;
    Table(PyObject *seq, const at::TensorBase &like) {
        require(PyList_CheckExact(seq) || PyTuple_CheckExact(seq));
        const Py_ssize_t count = PySequence_Fast_GET_SIZE(seq);
        require(count >= 1 && count <= kMaxTable);
        for (int i = 0; i < count; ++i) p[i] = dense(PySequence_Fast_GET_ITEM(seq, i), like, like.sizes(), true);
        for (; n < count; ++n) held[n] = Py_NewRef(PySequence_Fast_GET_ITEM(seq, n));
    }
    // Not where the thread is being taken down: it does not hold the lock then, and the process is ending.
    ~Table() {
        if (!PyGILState_Check()) return;
        while (n > 0) Py_DECREF(held[--n]);
    }
    Table(const Table &) = delete;
    Table &operator=(const Table &) = delete;
};

// The strided and two-shot forms launch without the interpreter lock, as they did through ctypes.  The plain
// forms keep it, as prepared calls do: whoever gives it up beside a thread that computes in Python waits a
// whole switch interval (5 ms) to have it back, 1000 times the call.
// Everything they pass has been read before the lock is given up: plain values only.
template <typename FN, typename... ARGS> astra_status_t unlocked(FN fn, ARGS... args) {
    static_assert((std::is_scalar_v<ARGS> && ...), "no object is looked at without the interpreter lock");
    PyThreadState *state = PyEval_SaveThread();
    const astra_status_t st = fn(args...);
    PyEval_RestoreThread(state);
    return st;
}

template <typename FN> FN entry(int kind) {
    require(astra_entry_points[kind] != nullptr);
    return reinterpret_cast<FN>(astra_entry_points[kind]);
}

template <typename CALL> PyObject *guarded(Py_ssize_t nargs, Py_ssize_t want, CALL call) {
    if (nargs != want) {
        PyErr_Format(PyExc_TypeError, "%zd arguments expected", want);
        return nullptr;
    }
    try {
        return PyLong_FromLong(static_cast<long>(call()));
    } catch (const Unusual &) {
    } catch (const std::exception &) {  // torch refused an access
    }
    // (Nothing else is caught: at the interpreter's end, a thread that comes for the lock again is unwound.)
    PyErr_Clear();  // the binding's own route decides
    Py_RETURN_NONE;
}

}  // namespace

extern "C" {

// rmsnorm(x, residual, weight, eps, stream)
PyObject *tc_rmsnorm(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 5, [&] {
        const at::TensorBase &x = tensor(a[0]);
        const astra_dtype_t dt = dtype_of(x);
        require(x.dim() == 2 && x.is_contiguous());
        const int64_t T = x.size(0), H = x.size(1), width[1] = {H};
        void *r = dense(a[1], x, x.sizes()), *w = dense(a[2], x, width);
        const float eps = number(a[3]);
        void *const stream = stream_of(a[4], x);
        void *const p_x = x.mutable_data_ptr();
        const auto fn = entry<decltype(&astra_fused_add_rmsnorm)>(KIND_RMSNORM);
        return fn(p_x, r, w, T, H, eps, dt, stream);
    });
}

// silu(out, input, stream)
PyObject *tc_silu(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 3, [&] {
        const at::TensorBase &in = tensor(a[1]);
        const astra_dtype_t dt = dtype_of(in);
        require(in.dim() == 2 && in.is_contiguous() && in.size(1) % 2 == 0);
        const int64_t T = in.size(0), D = in.size(1) / 2, sizes[2] = {T, D};
        void *out = dense(a[0], in, sizes);
        void *const stream = stream_of(a[2], in);
        void *const p_in = in.mutable_data_ptr();
        const auto fn = entry<decltype(&astra_silu_and_mul)>(KIND_SILU);
        return fn(out, p_in, T, D, dt, stream);
    });
}

// merge(v_out, lse_out, v_a, lse_a, v_b, lse_b, stream)
PyObject *tc_merge(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 7, [&] {
        const at::TensorBase &va = tensor(a[2]);
        const astra_dtype_t dt = dtype_of(va);
        require(va.dim() == 3 && va.is_contiguous());
        const int64_t T = va.size(0), Hh = va.size(1), D = va.size(2), sizes[2] = {T, Hh};
        void *vo = dense(a[0], va, va.sizes()), *vb = dense(a[4], va, va.sizes());
        void *so = a[1] == Py_None ? nullptr : scores(a[1], va, sizes);
        void *sa = scores(a[3], va, sizes), *sb = scores(a[5], va, sizes);
        void *const stream = stream_of(a[6], va);
        void *const p_va = va.mutable_data_ptr();
        const auto fn = entry<decltype(&astra_merge_attn_states_lse)>(KIND_MERGE);
        return fn(vo, static_cast<float *>(so), p_va, static_cast<float *>(sa), vb, static_cast<float *>(sb), T, Hh, D, dt, stream);
    });
}

// allreduce_rmsnorm(y, residual, parts, weight, eps, stream)
PyObject *tc_allreduce(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 6, [&] {
        const at::TensorBase &y = tensor(a[0]);
        const astra_dtype_t dt = dtype_of(y);
        require(y.dim() == 2 && y.is_contiguous());
        const int64_t T = y.size(0), H = y.size(1), width[1] = {H};
        void *r = dense(a[1], y, y.sizes()), *w = dense(a[3], y, width);
        const Table parts(a[2], y);
        const float eps = number(a[4]);
        void *const stream = stream_of(a[5], y);
        void *const p_y = y.mutable_data_ptr();
        const auto fn = entry<decltype(&astra_fused_allreduce_add_rmsnorm)>(KIND_ALLREDUCE_RMSNORM);
        return fn(p_y, r, parts.p, parts.n, w, T, H, eps, dt, stream);
    });
}

// allreduce_rmsnorm_ex(y_outs, residual_outs, residual, parts, weight, eps, stream)
PyObject *tc_allreduce_ex(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 7, [&] {
        const at::TensorBase &r = tensor(a[2]);
        const astra_dtype_t dt = dtype_of(r);
        require(r.dim() == 2 && r.is_contiguous());
        const int64_t T = r.size(0), H = r.size(1), width[1] = {H};
        void *w = dense(a[4], r, width);
        const Table parts(a[3], r), ys(a[0], r), rs(a[1], r);
        const float eps = number(a[5]);
        void *const stream = stream_of(a[6], r);
        void *const p_r = r.mutable_data_ptr();
        const auto fn = entry<decltype(&astra_fused_allreduce_add_rmsnorm_ex)>(KIND_ALLREDUCE_RMSNORM_EX);
        return unlocked(fn, ys.p, ys.n, rs.p, rs.n, p_r, parts.p, parts.n, w, T, H, eps, dt, stream);
    });
}

// rmsnorm_ex(y, residual_out, x, residual, weight, eps, stream)
PyObject *tc_rmsnorm_ex(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 7, [&] {
        const at::TensorBase &x = tensor(a[2]);
        const astra_dtype_t dt = dtype_of(x);
        require(x.dim() == 2);
        rows(a[2], x);
        const at::TensorBase &r = rows(a[3], x), &y = rows(a[0], x), &ro = rows(a[1], x);
        const int64_t T = x.size(0), H = x.size(1), width[1] = {H};
        void *w = dense(a[4], x, width);
        const float eps = number(a[5]);
        void *const stream = stream_of(a[6], x);
        void *const p_y = y.mutable_data_ptr();
        void *const p_ro = ro.mutable_data_ptr();
        void *const p_x = x.mutable_data_ptr();
        void *const p_r = r.mutable_data_ptr();
        const auto fn = entry<decltype(&astra_fused_add_rmsnorm_ex)>(KIND_RMSNORM_EX);
        return unlocked(fn, p_y, p_ro, p_x, p_r, w, T, H, pitch(y), pitch(ro), pitch(x), pitch(r), eps, dt, stream);
    });
}

// silu_ex(out, gate, up, stream)
PyObject *tc_silu_ex(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 4, [&] {
        const at::TensorBase &gate = tensor(a[1]);
        const astra_dtype_t dt = dtype_of(gate);
        require(gate.dim() == 2);
        rows(a[1], gate);
        const at::TensorBase &up = rows(a[2], gate), &out = rows(a[0], gate);
        void *const stream = stream_of(a[3], gate);
        void *const p_out = out.mutable_data_ptr();
        void *const p_gate = gate.mutable_data_ptr();
        void *const p_up = up.mutable_data_ptr();
        const auto fn = entry<decltype(&astra_silu_and_mul_ex)>(KIND_SILU_EX);
        return unlocked(fn, p_out, p_gate, p_up, gate.size(0), gate.size(1), pitch(out), pitch(gate), pitch(up), dt, stream);
    });
}

// merge_ex(v_out, lse_out, v_a, lse_a, v_b, lse_b, stream)
PyObject *tc_merge_ex(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 7, [&] {
        const at::TensorBase &va = tensor(a[2]);
        const astra_dtype_t dt = dtype_of(va);
        require(va.dim() == 3);
        rows(a[2], va);
        const at::TensorBase &vb = rows(a[4], va), &vo = rows(a[0], va);
        const int64_t T = va.size(0), Hh = va.size(1), D = va.size(2), sizes[2] = {T, Hh};
        int64_t st[12] = {va.stride(0), va.stride(1), vb.stride(0), vb.stride(1), vo.stride(0), vo.stride(1)};
        void *score[3] = {nullptr, nullptr, nullptr};
        PyObject *const given[3] = {a[3], a[5], a[1]};
        for (int i = 0; i < 3; ++i) {
            if (i == 2 && given[i] == Py_None) continue;
            const at::TensorBase &s = tensor(given[i]);
            require(s.scalar_type() == at::kFloat && s.sizes() == at::IntArrayRef(sizes) && s.device() == va.device());
            st[6 + 2 * i] = s.stride(0);
            st[7 + 2 * i] = s.stride(1);
            score[i] = s.mutable_data_ptr();
        }
        void *const stream = stream_of(a[6], va);
        void *const p_vo = vo.mutable_data_ptr();
        void *const p_va = va.mutable_data_ptr();
        void *const p_vb = vb.mutable_data_ptr();
        const auto fn = entry<decltype(&astra_merge_attn_states_lse_ex)>(KIND_MERGE_EX);
        return unlocked(fn, p_vo, static_cast<float *>(score[2]), p_va, static_cast<float *>(score[0]), p_vb,
                        static_cast<float *>(score[1]), T, Hh, D, st, dt, stream);
    });
}

// The torch release this file was compiled against; the build script finds it in the built file.
__attribute__((used)) const char astra_torch_marker[] = "astra-torch:" ASTRA_TORCH_VERSION ";";

}  // extern "C"
