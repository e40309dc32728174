/*
 * _astra_fastcall -- a CPython extension that re-issues prepared calls of the astra.h ABI.
 *
 * The Python binding reaches libastra.so through ctypes, whose per-call cost (about 1 us: argument
 * conversion and the foreign-function transition) is as large as the device time of the decode-sized
 * shapes of the paper's Table 4.  A prepared call has already validated and converted its arguments
 * once; this module keeps them in a C struct and `launch(prepared, stream)` passes them straight to
 * the entry point.  It only marshals: every argument check of the C ABI still runs inside the entry
 * point on every launch, and nothing is computed here.
 *
 * Direct calls on tensors are in torchcall.cpp, an extension of its own: it belongs to one torch release,
 * this one to none.
 *
 * The module does not link against libastra.so.  The binding hands it the addresses of the entry
 * points it has already resolved (`bind`), so there is one copy of the library in the process and
 * the staleness check made when the library was loaded covers these calls too.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include "astra.h"
#include "call_runs.h"
#include "fastcall.h"

#ifndef ASTRA_BUILD_ID
#define ASTRA_BUILD_ID "unidentified"
#endif
/* hash of the sources this module was compiled from; the build script finds it in the file */
__attribute__((used, visibility("default"))) const char astra_fastcall_build_marker[] =
    "astra-build-id:" ASTRA_BUILD_ID;

#define MAX_PARTS 16

typedef astra_status_t (*rmsnorm_fn)(void *, void *, const void *, int64_t, int64_t, float, astra_dtype_t, void *);
typedef astra_status_t (*silu_fn)(void *, const void *, int64_t, int64_t, astra_dtype_t, void *);
typedef astra_status_t (*merge_fn)(void *, float *, const void *, const float *, const void *, const float *,
                                   int64_t, int64_t, int64_t, astra_dtype_t, void *);
typedef astra_status_t (*allreduce_fn)(void *, void *, const void *const *, int32_t, const void *, int64_t,
                                       int64_t, float, astra_dtype_t, void *);

typedef astra_status_t (*run_fn)(int, int32_t, const astra_run_call *, const int64_t *, float, astra_dtype_t, void *);

static void *entry_points[KIND_PREPARED];
static run_fn issue_run;

typedef struct {
    PyObject_HEAD
    int kind;
    int dtype;
    int n_parts;
    float eps;
    void *ptr[6];               /* the call's pointer arguments, in the order of its declaration */
    int64_t ext[3];             /* the call's extents, in the order of its declaration */
    const void *parts[MAX_PARTS];
} Prepared;

static PyTypeObject PreparedType = {
    PyVarObject_HEAD_INIT(NULL, 0)
    .tp_name = "_astra_fastcall.Prepared",
    .tp_basicsize = sizeof(Prepared),
    .tp_flags = Py_TPFLAGS_DEFAULT,
    .tp_doc = "arguments of one astra call, ready to be launched",
};

static int as_address(PyObject *o, void **out) {
    if (o == Py_None) {
        *out = NULL;
        return 0;
    }
    *out = PyLong_AsVoidPtr(o);
    return (*out == NULL && PyErr_Occurred()) ? -1 : 0;
}

/* bind(kind, address): the entry point that calls of this kind go to */
static PyObject *fc_bind(PyObject *self, PyObject *args) {
    int kind;
    PyObject *addr;
    if (!PyArg_ParseTuple(args, "iO", &kind, &addr)) return NULL;
    if (kind < 0 || kind >= KIND_PREPARED) {
        PyErr_SetString(PyExc_ValueError, "unknown kind of call");
        return NULL;
    }
    void *p;
    if (as_address(addr, &p) < 0) return NULL;
    entry_points[kind] = p;
    Py_RETURN_NONE;
}

/* prepare(kind, pointers, extents, eps, dtype, parts) -> Prepared
 * pointers: the call's pointer arguments (ints or None) in declaration order; extents: its int64
 * extents in declaration order; parts: the partial hidden states of the all-reduce form (else ()). */
static PyObject *fc_prepare(PyObject *self, PyObject *args) {
    int kind, dtype;
    double eps;
    PyObject *pointers, *extents, *parts;
    if (!PyArg_ParseTuple(args, "iO!O!diO!", &kind, &PyTuple_Type, &pointers, &PyTuple_Type, &extents, &eps,
                          &dtype, &PyTuple_Type, &parts))
        return NULL;
    static const int n_pointers[KIND_PREPARED] = {3, 2, 6, 3};
    static const int n_extents[KIND_PREPARED] = {2, 2, 3, 2};
    if (kind < 0 || kind >= KIND_PREPARED) {
        PyErr_SetString(PyExc_ValueError, "unknown kind of call");
        return NULL;
    }
    if (entry_points[kind] == NULL) {
        PyErr_SetString(PyExc_RuntimeError, "no entry point bound for this kind of call");
        return NULL;
    }
    if (PyTuple_GET_SIZE(pointers) != n_pointers[kind] || PyTuple_GET_SIZE(extents) != n_extents[kind]) {
        PyErr_SetString(PyExc_ValueError, "wrong number of pointers or extents for this kind of call");
        return NULL;
    }
    const Py_ssize_t np = PyTuple_GET_SIZE(parts);
    if ((kind == KIND_ALLREDUCE_RMSNORM) ? (np < 1 || np > MAX_PARTS) : (np != 0)) {
        PyErr_SetString(PyExc_ValueError, "wrong number of partial hidden states");
        return NULL;
    }
    Prepared *p = PyObject_New(Prepared, &PreparedType);
    if (p == NULL) return NULL;
    p->kind = kind;
    p->dtype = dtype;
    p->eps = (float)eps;
    p->n_parts = (int)np;
    memset(p->ptr, 0, sizeof p->ptr);
    memset(p->ext, 0, sizeof p->ext);
    memset(p->parts, 0, sizeof p->parts);
    for (int i = 0; i < n_pointers[kind]; ++i)
        if (as_address(PyTuple_GET_ITEM(pointers, i), &p->ptr[i]) < 0) goto fail;
    for (int i = 0; i < n_extents[kind]; ++i) {
        p->ext[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(extents, i));
        if (p->ext[i] == -1 && PyErr_Occurred()) goto fail;
    }
    for (Py_ssize_t i = 0; i < np; ++i) {
        void *a;
        if (as_address(PyTuple_GET_ITEM(parts, i), &a) < 0) goto fail;
        p->parts[i] = a;
    }
    return (PyObject *)p;
fail:
    Py_DECREF(p);
    return NULL;
}

/* launch(prepared, stream_handle) -> status code of the entry point */
static PyObject *fc_launch(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
    if (nargs != 2 || !Py_IS_TYPE(args[0], &PreparedType)) {
        PyErr_SetString(PyExc_TypeError, "launch(prepared, stream_handle)");
        return NULL;
    }
    const Prepared *p = (const Prepared *)args[0];
    void *stream = PyLong_AsVoidPtr(args[1]);
    if (stream == NULL && PyErr_Occurred()) return NULL;
    const astra_dtype_t dt = (astra_dtype_t)p->dtype;
    void *fn = entry_points[p->kind];
    if (fn == NULL) {  /* unbound again since the call was prepared */
        PyErr_SetString(PyExc_RuntimeError, "no entry point bound for this kind of call");
        return NULL;
    }
    astra_status_t st;
    switch (p->kind) {
        case KIND_RMSNORM:
            st = ((rmsnorm_fn)fn)(p->ptr[0], p->ptr[1], p->ptr[2], p->ext[0], p->ext[1], p->eps, dt, stream);
            break;
        case KIND_SILU:
            st = ((silu_fn)fn)(p->ptr[0], p->ptr[1], p->ext[0], p->ext[1], dt, stream);
            break;
        case KIND_MERGE:
            st = ((merge_fn)fn)(p->ptr[0], (float *)p->ptr[1], p->ptr[2], (const float *)p->ptr[3], p->ptr[4],
                                (const float *)p->ptr[5], p->ext[0], p->ext[1], p->ext[2], dt, stream);
            break;
        default:
            st = ((allreduce_fn)fn)(p->ptr[0], p->ptr[1], p->parts, p->n_parts, p->ptr[2], p->ext[0], p->ext[1],
                                    p->eps, dt, stream);
            break;
    }
    return PyLong_FromLong((long)st);
}

/* bind_run(address): the library's astra_issue_run */
static PyObject *fc_bind_run(PyObject *self, PyObject *address) {
    void *p;
    if (as_address(address, &p) < 0) return NULL;
    issue_run = (run_fn)p;
    Py_RETURN_NONE;
}

/* Do two calls differ in nothing but their addresses?  (The all-reduce form is never part of a run.) */
static int alike(const Prepared *p, const Prepared *q) {
    return p->kind == q->kind && p->kind != KIND_ALLREDUCE_RMSNORM && p->dtype == q->dtype &&
           memcmp(&p->eps, &q->eps, sizeof p->eps) == 0 && memcmp(p->ext, q->ext, sizeof p->ext) == 0;
}

/* alike(prepared, prepared) -> whether the two can be in one run */
static PyObject *fc_alike(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
    if (nargs != 2 || !Py_IS_TYPE(args[0], &PreparedType) || !Py_IS_TYPE(args[1], &PreparedType)) {
        PyErr_SetString(PyExc_TypeError, "alike(prepared, prepared)");
        return NULL;
    }
    return PyBool_FromLong(alike((const Prepared *)args[0], (const Prepared *)args[1]));
}

/* launch_run(calls, stream_handle) -> status: calls that are alike, in order, in as few launches as their operands allow */
static PyObject *fc_launch_run(PyObject *self, PyObject *args) {
    PyObject *calls, *handle;
    void *stream;
    if (!PyArg_ParseTuple(args, "O!O", &PyList_Type, &calls, &handle) || as_address(handle, &stream) < 0) return NULL;
    const Py_ssize_t n = PyList_GET_SIZE(calls);
    if (n < 1 || n > INT32_MAX || issue_run == NULL) {
        PyErr_SetString(PyExc_ValueError, issue_run == NULL ? "no entry point bound for runs" : "no calls");
        return NULL;
    }
    astra_run_call *each = PyMem_Malloc((size_t)n * sizeof *each);
    if (each == NULL) return PyErr_NoMemory();
    const Prepared *first = (const Prepared *)PyList_GET_ITEM(calls, 0);
    for (Py_ssize_t i = 0; i < n; ++i) {
        PyObject *c = PyList_GET_ITEM(calls, i);
        if (!Py_IS_TYPE(c, &PreparedType) || !alike(first, (const Prepared *)c)) {
            PyMem_Free(each);
            PyErr_SetString(PyExc_ValueError, "the calls of a run are alike");
            return NULL;
        }
        memcpy(each[i].ptr, ((const Prepared *)c)->ptr, sizeof each[i].ptr);
    }
    const astra_status_t st = issue_run(first->kind, (int32_t)n, each, first->ext, first->eps, (astra_dtype_t)first->dtype, stream);
    PyMem_Free(each);
    return PyLong_FromLong((long)st);
}

/* The memory a call reads and writes: at most 6 + MAX_PARTS ranges, the first *written of them outputs. */
static int footprint_of(const Prepared *p, const void **at, int64_t *bytes, int *written) {
    const int64_t elem = p->dtype == ASTRA_FP32 ? 4 : 2;
    const int64_t all = p->ext[0] * p->ext[1] * elem, row = p->ext[1] * elem;
    int n;
    for (int i = 0; i < 6; ++i) at[i] = p->ptr[i];
    *written = 2;
    switch (p->kind) {
        case KIND_SILU:
            n = 2, *written = 1, bytes[0] = all, bytes[1] = 2 * all;
            break;
        case KIND_MERGE:
            n = 6, bytes[0] = bytes[2] = bytes[4] = all * p->ext[2], bytes[1] = bytes[3] = bytes[5] = p->ext[0] * p->ext[1] * 4;
            break;
        default:  /* the two norms; the all-reduce form has its partials besides */
            n = 3, bytes[0] = bytes[1] = all, bytes[2] = row;
            for (int i = 0; i < p->n_parts; ++i) at[n] = p->parts[i], bytes[n++] = all;
            break;
    }
    for (int i = 0; i < n; ++i)
        if (at[i] == NULL) bytes[i] = 0;
    return n;
}

/* footprint(prepared) -> ((address, bytes, is_written), ...): the memory the call reads and writes */
static PyObject *fc_footprint(PyObject *self, PyObject *arg) {
    if (!Py_IS_TYPE(arg, &PreparedType)) {
        PyErr_SetString(PyExc_TypeError, "footprint(prepared)");
        return NULL;
    }
    const void *at[6 + MAX_PARTS];
    int64_t bytes[6 + MAX_PARTS];
    int written;
    const int n = footprint_of((const Prepared *)arg, at, bytes, &written);
    PyObject *out = PyTuple_New(n);
    for (int i = 0; out != NULL && i < n; ++i) {
        PyObject *item = Py_BuildValue("(KLi)", (unsigned long long)(uintptr_t)at[i], (long long)bytes[i], i < written);
        if (item == NULL) Py_CLEAR(out);
        else PyTuple_SET_ITEM(out, i, item);
    }
    return out;
}

/* ---- which calls of a sequence depend on one another ------------------------------------------------------ */

typedef struct {
    uint64_t begin, end;
    int call, written;
} Range;

static int by_address(const void *a, const void *b) {
    const Range *p = a, *q = b;
    if (p->begin != q->begin) return p->begin < q->begin ? -1 : 1;
    return (p->end > q->end) - (p->end < q->end);
}

static int root_of(int *parent, int i) {
    while (parent[i] != i) i = parent[i] = parent[parent[i]];
    return i;
}

/* Groups (0, 1, ... in order of first appearance, into group[n_calls]) such that two calls of different groups share
 * no byte that either of them writes.  One sweep in address order: a range that reaches into the present run of
 * overlapping written ranges joins the run's call; a read in front of a run waits until the run begins. */
static int group_calls(Range *r, Py_ssize_t n, int *group, Py_ssize_t n_calls) {
    int *parent = PyMem_Malloc((size_t)(2 * n_calls + 1) * sizeof(int));
    Range *reads = PyMem_Malloc((size_t)(n + 1) * sizeof(Range));  /* reads that may reach a later run */
    if (parent == NULL || reads == NULL) {
        PyMem_Free(parent);
        PyMem_Free(reads);
        return -1;
    }
    int *number = parent + n_calls;
    for (int i = 0; i < n_calls; ++i) parent[i] = i, number[i] = -1;
    uint64_t run_end = 0;
    int owner = -1;
    Py_ssize_t n_reads = 0;
    for (Py_ssize_t i = 0; i < n; ++i) {
        const int in_run = owner >= 0 && r[i].begin < run_end;
        if (in_run) parent[root_of(parent, r[i].call)] = root_of(parent, owner);
        if (!r[i].written) {
            reads[n_reads++] = r[i];
            continue;
        }
        if (!in_run) owner = r[i].call, run_end = r[i].end;
        else if (r[i].end > run_end) run_end = r[i].end;
        /* the reads that reach into this range are of its group from here on: one stands for all */
        uint64_t reach = 0;
        for (Py_ssize_t k = 0; k < n_reads; ++k) {
            if (reads[k].end <= r[i].begin) continue;  /* ends before this and every later written range */
            parent[root_of(parent, reads[k].call)] = root_of(parent, r[i].call);
            if (reads[k].end > reach) reach = reads[k].end;
        }
        n_reads = reach > 0;
        reads[0] = (Range){r[i].begin, reach, r[i].call, 0};
    }
    int next = 0;
    for (int i = 0; i < n_calls; ++i) {
        const int g = root_of(parent, i);
        if (number[g] < 0) number[g] = next++;
        group[i] = number[g];
    }
    PyMem_Free(parent);
    PyMem_Free(reads);
    return 0;
}

static PyObject *as_list(const int *v, Py_ssize_t n) {
    PyObject *out = PyList_New(n);
    for (Py_ssize_t i = 0; out != NULL && i < n; ++i) {
        PyObject *item = PyLong_FromLong(v[i]);
        if (item == NULL) Py_CLEAR(out);
        else PyList_SET_ITEM(out, i, item);
    }
    return out;
}

/* The ranges of a sequence of calls; a call is a Prepared, or the ((address, bytes, is_written), ...) of one.
 * Returns the number of calls, or -1 with an exception set; *r is the caller's to free. */
static Py_ssize_t gather(PyObject *arg, Range **r, Py_ssize_t *n) {
    PyObject *calls = PySequence_Fast(arg, "a sequence of calls");
    if (calls == NULL) return -1;
    const Py_ssize_t n_calls = PySequence_Fast_GET_SIZE(calls);
    Py_ssize_t room = 0, done = -1;
    *r = NULL, *n = 0;
    for (Py_ssize_t c = 0; c < n_calls; ++c) {
        PyObject *call = PySequence_Fast_GET_ITEM(calls, c), *given = NULL;
        const void *at[6 + MAX_PARTS];
        int64_t bytes[6 + MAX_PARTS];
        int written = 0;
        Py_ssize_t count;
        if (Py_IS_TYPE(call, &PreparedType)) {
            count = footprint_of((const Prepared *)call, at, bytes, &written);
        } else {
            if ((given = PySequence_Fast(call, "a prepared call or its footprint")) == NULL) goto out;
            count = PySequence_Fast_GET_SIZE(given);
        }
        if (*n + count > room) {
            room = 2 * (*n + count) + 4 * (n_calls - c);
            Range *more = PyMem_Realloc(*r, (size_t)room * sizeof(Range));
            if (more == NULL) {
                Py_XDECREF(given);
                PyErr_NoMemory();
                goto out;
            }
            *r = more;
        }
        for (Py_ssize_t i = 0; i < count; ++i) {
            unsigned long long begin;
            long long size;
            int is_written;
            if (given == NULL) {
                begin = (unsigned long long)(uintptr_t)at[i], size = bytes[i], is_written = i < written;
            } else if (!PyArg_ParseTuple(PySequence_Fast_GET_ITEM(given, i), "KLp", &begin, &size, &is_written)) {
                Py_DECREF(given);
                goto out;
            }
            if (size > 0) (*r)[(*n)++] = (Range){begin, begin + (uint64_t)size, (int)c, is_written};
        }
        Py_XDECREF(given);
    }
    if (*n > 0) qsort(*r, (size_t)*n, sizeof(Range), by_address);
    done = n_calls;
out:
    Py_DECREF(calls);
    return done;
}

/* independent_groups(calls) -> group number of each call */
static PyObject *fc_independent_groups(PyObject *self, PyObject *arg) {
    Range *r = NULL;
    Py_ssize_t n;
    const Py_ssize_t n_calls = gather(arg, &r, &n);
    PyObject *out = NULL;
    if (n_calls >= 0) {
        int *group = PyMem_Malloc((size_t)(n_calls + 1) * sizeof(int));
        if (group == NULL || group_calls(r, n, group, n_calls) < 0) PyErr_NoMemory();
        else out = as_list(group, n_calls);
        PyMem_Free(group);
    }
    PyMem_Free(r);
    return out;
}

/* one_address_each(calls, query) -> whether every range lies in memory that has one address in this process.
 * `query` is the address of the driver's cuPointerGetAttributes.  Memory of the plain allocators (those whose
 * memory can be handed to another process as a whole) cannot be mapped a second time here; physical memory that
 * was mapped by hand, imported memory and host memory can. */
typedef int (*attributes_fn)(unsigned, int *, void **, unsigned long long);

static PyObject *fc_one_address_each(PyObject *self, PyObject *args) {
    PyObject *calls, *address;
    if (!PyArg_ParseTuple(args, "OO", &calls, &address)) return NULL;
    void *p;
    if (as_address(address, &p) < 0) return NULL;
    const attributes_fn query = (attributes_fn)p;
    Range *r = NULL;
    Py_ssize_t n;
    if (gather(calls, &r, &n) < 0) {
        PyMem_Free(r);
        return NULL;
    }
    /* CU_POINTER_ATTRIBUTE_IS_LEGACY_CUDA_IPC_CAPABLE, _RANGE_START_ADDR, _RANGE_SIZE */
    int wanted[3] = {10, 11, 12}, sole = query != NULL;
    uint64_t known = 0;  /* ranges that end at or before it and begin after the allocation's start are known */
    for (Py_ssize_t i = 0; sole && i < n; ++i) {
        if (r[i].end <= known) continue;
        uint64_t plain = 0, start = 0, size = 0;
        void *out[3] = {&plain, &start, &size};
        sole = query(3, wanted, out, r[i].begin) == 0 && (plain & 0xff) != 0 && start <= r[i].begin &&
               r[i].end <= start + size;
        known = start + size;
    }
    PyMem_Free(r);
    return PyBool_FromLong(sole);
}

static PyObject *fc_build_id(PyObject *self, PyObject *noargs) {
    return PyUnicode_FromString(astra_fastcall_build_marker + sizeof("astra-build-id:") - 1);
}

static PyMethodDef methods[] = {
    {"bind", fc_bind, METH_VARARGS, "bind(kind, address): set the entry point of one kind of call"},
    {"prepare", fc_prepare, METH_VARARGS, "prepare(kind, pointers, extents, eps, dtype, parts) -> Prepared"},
    {"launch", (PyCFunction)(void (*)(void))fc_launch, METH_FASTCALL, "launch(prepared, stream_handle) -> status"},
    {"bind_run", fc_bind_run, METH_O, "bind_run(address): set the entry point of runs of calls"},
    {"alike", (PyCFunction)(void (*)(void))fc_alike, METH_FASTCALL, "alike(prepared, prepared) -> whether the two can be in one run"},
    {"launch_run", fc_launch_run, METH_VARARGS, "launch_run(calls, stream_handle) -> status of the calls, issued in order"},
    {"footprint", fc_footprint, METH_O, "footprint(prepared) -> ((address, bytes, is_written), ...)"},
    {"independent_groups", fc_independent_groups, METH_O, "independent_groups(calls) -> group number of each call"},
    {"one_address_each", fc_one_address_each, METH_VARARGS,
     "one_address_each(calls, query) -> whether all their memory has one address in this process"},
    {"build_id", fc_build_id, METH_NOARGS, "hash of the sources this module was compiled from"},
    {NULL, NULL, 0, NULL},
};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_astra_fastcall",
                                    "re-issue prepared calls of the astra C ABI without ctypes", -1, methods};

PyMODINIT_FUNC PyInit__astra_fastcall(void) {
    if (PyType_Ready(&PreparedType) < 0) return NULL;
    PyObject *m = PyModule_Create(&module);
    if (m == NULL) return NULL;
    Py_INCREF(&PreparedType);
    if (PyModule_AddObject(m, "Prepared", (PyObject *)&PreparedType) < 0) {
        Py_DECREF(&PreparedType);
        Py_DECREF(m);
        return NULL;
    }
    PyModule_AddIntConstant(m, "KIND_RMSNORM", KIND_RMSNORM);
    PyModule_AddIntConstant(m, "KIND_SILU", KIND_SILU);
    PyModule_AddIntConstant(m, "KIND_MERGE", KIND_MERGE);
    PyModule_AddIntConstant(m, "KIND_ALLREDUCE_RMSNORM", KIND_ALLREDUCE_RMSNORM);
    return m;
}
