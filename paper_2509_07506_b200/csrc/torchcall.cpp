// _astra_torchcall -- a CPython extension for direct calls of the astra.h ABI on torch tensors, without
// Python-level checks.  It reads torch's C++ objects and so belongs to one torch release; with another one the
// binding leaves it unloaded and takes its own route.
//
// A direct call from the binding's Python code costs 3.5 to 12 us of attribute reads, checks and argument
// conversions, more than the launch and far more than the kernel of a decode-sized shape.  Each function
// here makes the same checks on the tensors' C++ objects and hands addresses and the current stream to the
// entry point.  It answers the ordinary case only: whenever a check does not hold, or anything about an
// operand is unusual (a tensor subclass, a functorch or functionalisation wrapper, an active torch-function
// mode, another current device), it returns None without having launched anything, and the binding takes
// its own route, which launches or raises the precise error.  Otherwise it returns the entry point's status;
// every argument check of the C ABI still runs there.
// Host time per call, enqueued back to back, Python-level checks -> here (nearly all of it the launch): rmsnorm 5.5 ->
// 2.2 us, silu 5.3 -> 2.0, merge 7.9 -> 2.2, all-reduce with 8 partials 11.9 -> 2.5; the strided forms of norm and merge 12.4 ->
// 2.2 and 15.7 -> 2.3, and 26.6 -> 3.1 us with 8 partials and 8 destinations.
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

#ifndef ASTRA_BUILD_ID
#define ASTRA_BUILD_ID "unidentified"
#endif

namespace {

constexpr int kMaxTable = 16;

void *entry_points[KIND_COUNT];

// What a call that is not the ordinary case answers instead of a status.  (A value and not an exception: such
// calls go on to the Python route on every call, 12 us for a generator of partials, and a C++ exception adds 2.)
constexpr int kUnusual = -1;

const at::TensorBase *tensor(PyObject *o) {
    if (!THPVariable_CheckExact(o)) return nullptr;  // Tensor or Parameter, no subclass
    const at::TensorBase &t = THPVariable_Unpack(o);
    static const c10::DispatchKeySet wrappers({c10::DispatchKey::Python, c10::DispatchKey::Functionalize,
                                               c10::DispatchKey::FuncTorchBatched, c10::DispatchKey::FuncTorchGradWrapper,
                                               c10::DispatchKey::Batched, c10::DispatchKey::Negative,
                                               c10::DispatchKey::Conjugate, c10::DispatchKey::ZeroTensor});
    if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || !t.has_storage() || t.key_set().has_any(wrappers))
        return nullptr;
    return &t;
}

bool dtype_of(const at::TensorBase &t, astra_dtype_t *dt) {
    switch (t.scalar_type()) {
        case at::kBFloat16: *dt = ASTRA_BF16; return true;
        case at::kHalf: *dt = ASTRA_FP16; return true;
        case at::kFloat: *dt = ASTRA_FP32; return true;
        default: return false;
    }
}

// The call's leading operand: its tensor and storage type.
const at::TensorBase *leading(PyObject *o, int64_t dims, bool contiguous, astra_dtype_t *dt) {
    const at::TensorBase *t = tensor(o);
    return t && dtype_of(*t, dt) && t->dim() == dims && (!contiguous || t->is_contiguous()) ? t : nullptr;
}

// Same dtype and shape as `like`, contiguous, on its device (unless it may be a peer's).
bool dense(PyObject *o, const at::TensorBase &like, at::IntArrayRef sizes, void **p, bool any_device = false) {
    const at::TensorBase *t = tensor(o);
    if (!t || t->scalar_type() != like.scalar_type() || t->sizes() != sizes || !t->is_contiguous() ||
        (!any_device && t->device() != like.device()))
        return false;
    *p = t->mutable_data_ptr();
    return true;
}

bool scores(PyObject *o, const at::TensorBase &like, at::IntArrayRef sizes, float **p) {
    const at::TensorBase *t = tensor(o);
    if (!t || t->scalar_type() != at::kFloat || t->sizes() != sizes || !t->is_contiguous() || t->device() != like.device())
        return false;
    *p = static_cast<float *>(t->mutable_data_ptr());
    return true;
}

// Same dtype, shape and device as `like`, innermost dimension contiguous.
const at::TensorBase *rows(PyObject *o, const at::TensorBase &like) {
    const at::TensorBase *t = tensor(o);
    return t && t->scalar_type() == like.scalar_type() && t->sizes() == like.sizes() && t->device() == like.device() &&
                   (t->size(-1) <= 1 || t->stride(-1) == 1)
               ? t
               : nullptr;
}

// A single row may report any stride; its width is used then.
int64_t pitch(const at::TensorBase &t) {
    return t.size(0) > 1 ? t.stride(0) : std::max<int64_t>(t.stride(0), t.size(1));
}

bool number(PyObject *o, float *out) {
    if (!PyFloat_Check(o) && !PyLong_CheckExact(o)) return false;
    const double v = PyFloat_AsDouble(o);
    *out = static_cast<float>(v);
    return !(v == -1.0 && PyErr_Occurred());
}

// The stream to launch on; the call's device must be current, since the C side launches on that one.
bool stream_of(PyObject *stream, const at::TensorBase &t, void **out) {
    const c10::DeviceIndex dev = t.device().index();
    if (at::impl::torch_function_mode_enabled() || dev != c10::cuda::current_device()) return false;
    if (stream == Py_None) {
        *out = c10::cuda::getCurrentCUDAStream(dev).stream();
        return true;
    }
    PyObject *handle = PyObject_GetAttrString(stream, "cuda_stream");
    if (handle == nullptr) return false;
    *out = PyLong_Check(handle) ? PyLong_AsVoidPtr(handle) : nullptr;
    const bool known = PyLong_Check(handle) && !PyErr_Occurred();
    Py_DECREF(handle);
    return known;
}

// Addresses of 1 to 16 dense tensors in a list or tuple; they may live on other GPUs.
// The table holds references: a list may be changed by another thread while the call runs unlocked.
struct Table {
    void *p[kMaxTable];
    PyObject *held[kMaxTable];
    int n = 0;
    Table() = default;
    bool fill(PyObject *seq, const at::TensorBase &like) {
        if (!PyList_CheckExact(seq) && !PyTuple_CheckExact(seq)) return false;
        const Py_ssize_t count = PySequence_Fast_GET_SIZE(seq);
        if (count < 1 || count > kMaxTable) return false;
        for (int i = 0; i < count; ++i)
            if (!dense(PySequence_Fast_GET_ITEM(seq, i), like, like.sizes(), &p[i], true)) return false;
        for (; n < count; ++n) held[n] = Py_NewRef(PySequence_Fast_GET_ITEM(seq, n));
        return true;
    }
    // Not where the thread is being taken down: it does not hold the lock then, and the process is ending.
    ~Table() {
        if (n == 0 || !PyGILState_Check()) return;
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

// The entry point of one kind of call, or null where none is bound.
template <typename FN> FN entry(int kind) { return reinterpret_cast<FN>(entry_points[kind]); }

template <typename CALL> PyObject *guarded(Py_ssize_t nargs, Py_ssize_t want, CALL call) {
    if (nargs != want) {
        PyErr_Format(PyExc_TypeError, "%zd arguments expected", want);
        return nullptr;
    }
    int st = kUnusual;
    try {
        st = call();
    } catch (const std::exception &) {  // torch refused an access
    }
    // (Nothing else is caught: at the interpreter's end, a thread that comes for the lock again is unwound.)
    if (st != kUnusual) return PyLong_FromLong(st);
    PyErr_Clear();  // the binding's own route decides
    Py_RETURN_NONE;
}

// rmsnorm(x, residual, weight, eps, stream)
PyObject *tc_rmsnorm(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 5, [&]() -> int {
        astra_dtype_t dt;
        const at::TensorBase *x = leading(a[0], 2, true, &dt);
        const auto fn = entry<decltype(&astra_fused_add_rmsnorm)>(KIND_RMSNORM);
        if (!x || !fn) return kUnusual;
        const int64_t T = x->size(0), H = x->size(1), width[1] = {H};
        void *r, *w, *stream;
        float eps;
        if (!dense(a[1], *x, x->sizes(), &r) || !dense(a[2], *x, width, &w) || !number(a[3], &eps) ||
            !stream_of(a[4], *x, &stream))
            return kUnusual;
        return fn(x->mutable_data_ptr(), r, w, T, H, eps, dt, stream);
    });
}

// silu(out, input, stream)
PyObject *tc_silu(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 3, [&]() -> int {
        astra_dtype_t dt;
        const at::TensorBase *in = leading(a[1], 2, true, &dt);
        const auto fn = entry<decltype(&astra_silu_and_mul)>(KIND_SILU);
        if (!in || !fn || in->size(1) % 2 != 0) return kUnusual;
        const int64_t T = in->size(0), D = in->size(1) / 2, sizes[2] = {T, D};
        void *out, *stream;
        if (!dense(a[0], *in, sizes, &out) || !stream_of(a[2], *in, &stream)) return kUnusual;
        return fn(out, in->mutable_data_ptr(), T, D, dt, stream);
    });
}

// merge(v_out, lse_out, v_a, lse_a, v_b, lse_b, stream)
PyObject *tc_merge(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 7, [&]() -> int {
        astra_dtype_t dt;
        const at::TensorBase *va = leading(a[2], 3, true, &dt);
        const auto fn = entry<decltype(&astra_merge_attn_states_lse)>(KIND_MERGE);
        if (!va || !fn) return kUnusual;
        const int64_t T = va->size(0), Hh = va->size(1), D = va->size(2), sizes[2] = {T, Hh};
        void *vo, *vb, *stream;
        float *so = nullptr, *sa, *sb;
        if (!dense(a[0], *va, va->sizes(), &vo) || !dense(a[4], *va, va->sizes(), &vb) ||
            (a[1] != Py_None && !scores(a[1], *va, sizes, &so)) || !scores(a[3], *va, sizes, &sa) ||
            !scores(a[5], *va, sizes, &sb) || !stream_of(a[6], *va, &stream))
            return kUnusual;
        return fn(vo, so, va->mutable_data_ptr(), sa, vb, sb, T, Hh, D, dt, stream);
    });
}

// allreduce_rmsnorm(y, residual, parts, weight, eps, stream)
PyObject *tc_allreduce(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 6, [&]() -> int {
        astra_dtype_t dt;
        const at::TensorBase *y = leading(a[0], 2, true, &dt);
        const auto fn = entry<decltype(&astra_fused_allreduce_add_rmsnorm)>(KIND_ALLREDUCE_RMSNORM);
        if (!y || !fn) return kUnusual;
        const int64_t T = y->size(0), H = y->size(1), width[1] = {H};
        void *r, *w, *stream;
        float eps;
        Table parts;
        if (!dense(a[1], *y, y->sizes(), &r) || !dense(a[3], *y, width, &w) || !parts.fill(a[2], *y) ||
            !number(a[4], &eps) || !stream_of(a[5], *y, &stream))
            return kUnusual;
        return fn(y->mutable_data_ptr(), r, parts.p, parts.n, w, T, H, eps, dt, stream);
    });
}

// allreduce_rmsnorm_ex(y_outs, residual_outs, residual, parts, weight, eps, stream)
PyObject *tc_allreduce_ex(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 7, [&]() -> int {
        astra_dtype_t dt;
        const at::TensorBase *r = leading(a[2], 2, true, &dt);
        const auto fn = entry<decltype(&astra_fused_allreduce_add_rmsnorm_ex)>(KIND_ALLREDUCE_RMSNORM_EX);
        if (!r || !fn) return kUnusual;
        const int64_t T = r->size(0), H = r->size(1), width[1] = {H};
        void *w, *stream;
        float eps;
        Table parts, ys, rs;
        if (!dense(a[4], *r, width, &w) || !parts.fill(a[3], *r) || !ys.fill(a[0], *r) || !rs.fill(a[1], *r) ||
            !number(a[5], &eps) || !stream_of(a[6], *r, &stream))
            return kUnusual;
        return unlocked(fn, ys.p, ys.n, rs.p, rs.n, r->mutable_data_ptr(), parts.p, parts.n, w, T, H, eps, dt, stream);
    });
}

// rmsnorm_ex(y, residual_out, x, residual, weight, eps, stream)
PyObject *tc_rmsnorm_ex(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 7, [&]() -> int {
        astra_dtype_t dt;
        const at::TensorBase *x = leading(a[2], 2, false, &dt);
        const auto fn = entry<decltype(&astra_fused_add_rmsnorm_ex)>(KIND_RMSNORM_EX);
        if (!x || !fn || !rows(a[2], *x)) return kUnusual;
        const at::TensorBase *r = rows(a[3], *x), *y = rows(a[0], *x), *ro = rows(a[1], *x);
        const int64_t T = x->size(0), H = x->size(1), width[1] = {H};
        void *w, *stream;
        float eps;
        if (!r || !y || !ro || !dense(a[4], *x, width, &w) || !number(a[5], &eps) || !stream_of(a[6], *x, &stream))
            return kUnusual;
        return unlocked(fn, y->mutable_data_ptr(), ro->mutable_data_ptr(), x->mutable_data_ptr(), r->mutable_data_ptr(), w,
                        T, H, pitch(*y), pitch(*ro), pitch(*x), pitch(*r), eps, dt, stream);
    });
}

// silu_ex(out, gate, up, stream)
PyObject *tc_silu_ex(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 4, [&]() -> int {
        astra_dtype_t dt;
        const at::TensorBase *gate = leading(a[1], 2, false, &dt);
        const auto fn = entry<decltype(&astra_silu_and_mul_ex)>(KIND_SILU_EX);
        if (!gate || !fn || !rows(a[1], *gate)) return kUnusual;
        const at::TensorBase *up = rows(a[2], *gate), *out = rows(a[0], *gate);
        void *stream;
        if (!up || !out || !stream_of(a[3], *gate, &stream)) return kUnusual;
        return unlocked(fn, out->mutable_data_ptr(), gate->mutable_data_ptr(), up->mutable_data_ptr(), gate->size(0),
                        gate->size(1), pitch(*out), pitch(*gate), pitch(*up), dt, stream);
    });
}

// merge_ex(v_out, lse_out, v_a, lse_a, v_b, lse_b, stream)
PyObject *tc_merge_ex(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded(nargs, 7, [&]() -> int {
        astra_dtype_t dt;
        const at::TensorBase *va = leading(a[2], 3, false, &dt);
        const auto fn = entry<decltype(&astra_merge_attn_states_lse_ex)>(KIND_MERGE_EX);
        if (!va || !fn || !rows(a[2], *va)) return kUnusual;
        const at::TensorBase *vb = rows(a[4], *va), *vo = rows(a[0], *va);
        if (!vb || !vo) return kUnusual;
        const int64_t T = va->size(0), Hh = va->size(1), D = va->size(2), sizes[2] = {T, Hh};
        int64_t st[12] = {va->stride(0), va->stride(1), vb->stride(0), vb->stride(1), vo->stride(0), vo->stride(1)};
        float *score[3] = {nullptr, nullptr, nullptr};
        PyObject *const given[3] = {a[3], a[5], a[1]};
        for (int i = 0; i < 3; ++i) {
            if (i == 2 && given[i] == Py_None) continue;
            const at::TensorBase *s = tensor(given[i]);
            if (!s || s->scalar_type() != at::kFloat || s->sizes() != at::IntArrayRef(sizes) || s->device() != va->device())
                return kUnusual;
            st[6 + 2 * i] = s->stride(0);
            st[7 + 2 * i] = s->stride(1);
            score[i] = static_cast<float *>(s->mutable_data_ptr());
        }
        void *stream;
        if (!stream_of(a[6], *va, &stream)) return kUnusual;
        return unlocked(fn, vo->mutable_data_ptr(), score[2], va->mutable_data_ptr(), score[0], vb->mutable_data_ptr(),
                        score[1], T, Hh, D, st, dt, stream);
    });
}

// What this file was compiled from and against; the build script and the binding find both in the built file.
__attribute__((used)) const char build_marker[] = "astra-build-id:" ASTRA_BUILD_ID;
__attribute__((used)) const char torch_marker[] = "astra-torch:" ASTRA_TORCH_VERSION ";";

PyObject *tc_build_id(PyObject *, PyObject *) {
    return PyUnicode_FromString(build_marker + sizeof("astra-build-id:") - 1);
}

// bind(kind, address): the entry point that calls of this kind go to
PyObject *tc_bind(PyObject *, PyObject *args) {
    int kind;
    PyObject *address;
    if (!PyArg_ParseTuple(args, "iO", &kind, &address)) return nullptr;
    if (kind < 0 || kind >= KIND_COUNT) {
        PyErr_SetString(PyExc_ValueError, "unknown kind of call");
        return nullptr;
    }
    void *p = address == Py_None ? nullptr : PyLong_AsVoidPtr(address);
    if (p == nullptr && PyErr_Occurred()) return nullptr;
    entry_points[kind] = p;
    Py_RETURN_NONE;
}

#define DIRECT(name, fn, doc) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL, doc " -> status, or None: not the ordinary case"}
PyMethodDef methods[] = {
    {"bind", tc_bind, METH_VARARGS, "bind(kind, address): set the entry point of one kind of call"},
    DIRECT("rmsnorm", tc_rmsnorm, "rmsnorm(x, residual, weight, eps, stream)"),
    DIRECT("silu", tc_silu, "silu(out, input, stream)"),
    DIRECT("merge", tc_merge, "merge(v_out, lse_out, v_a, lse_a, v_b, lse_b, stream)"),
    DIRECT("allreduce_rmsnorm", tc_allreduce, "allreduce_rmsnorm(y, residual, parts, weight, eps, stream)"),
    DIRECT("rmsnorm_ex", tc_rmsnorm_ex, "rmsnorm_ex(y, residual_out, x, residual, weight, eps, stream)"),
    DIRECT("silu_ex", tc_silu_ex, "silu_ex(out, gate, up, stream)"),
    DIRECT("merge_ex", tc_merge_ex, "merge_ex(v_out, lse_out, v_a, lse_a, v_b, lse_b, stream)"),
    DIRECT("allreduce_rmsnorm_ex", tc_allreduce_ex,
           "allreduce_rmsnorm_ex(y_outs, residual_outs, residual, parts, weight, eps, stream)"),
    {"build_id", tc_build_id, METH_NOARGS, "hash of the sources this module was compiled from"},
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_astra_torchcall", "direct calls of the astra C ABI on torch tensors", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__astra_torchcall(void) {
    PyObject *m = PyModule_Create(&module);
    if (m == nullptr) return nullptr;
    const struct { const char *name; int kind; } kinds[] = {
        {"KIND_RMSNORM", KIND_RMSNORM}, {"KIND_SILU", KIND_SILU}, {"KIND_MERGE", KIND_MERGE},
        {"KIND_ALLREDUCE_RMSNORM", KIND_ALLREDUCE_RMSNORM}, {"KIND_RMSNORM_EX", KIND_RMSNORM_EX},
        {"KIND_SILU_EX", KIND_SILU_EX}, {"KIND_MERGE_EX", KIND_MERGE_EX},
        {"KIND_ALLREDUCE_RMSNORM_EX", KIND_ALLREDUCE_RMSNORM_EX}};
    for (const auto &k : kinds) {
        if (PyModule_AddIntConstant(m, k.name, k.kind) < 0) {
            Py_DECREF(m);
            return nullptr;
        }
    }
    return m;
}
