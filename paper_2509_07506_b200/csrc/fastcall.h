/* Shared by the two halves of the _astra_fastcall extension (fastcall.c and torchcall.cpp). */
#pragma once

#include <Python.h>

enum {  /* the first KIND_PREPARED kinds can be prepared */
    KIND_RMSNORM = 0,
    KIND_SILU = 1,
    KIND_MERGE = 2,
    KIND_ALLREDUCE_RMSNORM = 3,
    KIND_PREPARED = 4,
    KIND_RMSNORM_EX = 4,
    KIND_SILU_EX = 5,
    KIND_MERGE_EX = 6,
    KIND_ALLREDUCE_RMSNORM_EX = 7,
    KIND_COUNT = 8
};

#ifdef __cplusplus
extern "C" {
#endif

extern void *astra_entry_points[KIND_COUNT];
extern const char astra_torch_marker[];  /* "astra-torch:<release>;" */

PyObject *tc_rmsnorm(PyObject *, PyObject *const *, Py_ssize_t);
PyObject *tc_silu(PyObject *, PyObject *const *, Py_ssize_t);
PyObject *tc_merge(PyObject *, PyObject *const *, Py_ssize_t);
PyObject *tc_allreduce(PyObject *, PyObject *const *, Py_ssize_t);
PyObject *tc_rmsnorm_ex(PyObject *, PyObject *const *, Py_ssize_t);
PyObject *tc_silu_ex(PyObject *, PyObject *const *, Py_ssize_t);
PyObject *tc_merge_ex(PyObject *, PyObject *const *, Py_ssize_t);
PyObject *tc_allreduce_ex(PyObject *, PyObject *const *, Py_ssize_t);

#ifdef __cplusplus
}
#endif
