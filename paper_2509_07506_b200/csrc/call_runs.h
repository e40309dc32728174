/* Issuing several prepared calls of one kind and shape at once: the interface between the library and the
 * _astra_fastcall extension.  Internal: not part of astra.h. */
#pragma once

#include "astra.h"

#ifdef __cplusplus
extern "C" {
#endif

enum { ASTRA_RUN_POINTERS = 6 };

/* One call's pointer arguments, in the order of its entry point's declaration. */
typedef struct {
    void *ptr[ASTRA_RUN_POINTERS];
} astra_run_call;

/*
 * The n calls one after the other, as if issued one by one through the entry point of their kind (KIND_RMSNORM,
 * KIND_SILU or KIND_MERGE of fastcall.h): every output bit for bit, except that the squares of a norm's row may
 * be summed in another order.  `ext`, eps and dtype are the same for all.  Consecutive calls whose operands allow
 * it share one launch; a call that the entry point refuses ends the run with that status, and those before it
 * are enqueued.
 */
astra_status_t astra_issue_run(int kind, int32_t n, const astra_run_call *calls, const int64_t *ext, float eps,
                               astra_dtype_t dtype, void *cuda_stream);

/*
 * The launches that astra_issue_run would make of these calls: their number, and how many calls each of them takes, in
 * order (room for n).  Nothing is launched, and no address is followed.
 */
astra_status_t astra_plan_run(int kind, int32_t n, const astra_run_call *calls, const int64_t *ext, astra_dtype_t dtype,
                              int32_t *counts, int32_t *launches);

#ifdef __cplusplus
}
#endif
