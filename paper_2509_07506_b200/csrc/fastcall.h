/* Kinds of calls, shared by the _astra_fastcall (fastcall.c) and _astra_torchcall (torchcall.cpp) extensions. */
#pragma once

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
