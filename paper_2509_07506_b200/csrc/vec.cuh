// Vector memory access and 16-bit storage conversion helpers shared by the three kernels.
//
// Every kernel here is HBM-bound: each input byte is read once and each output byte written once.
// The helpers therefore expose (a) the widest aligned global access the data allows (2, 4, 8, 16 or
// 32 bytes per thread; 32-byte accesses exist on sm_100 and later) with cache hints for once-touched
// data, and (b) exact widening / single-rounding narrowing between the storage types and binary32.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "astra.h"

namespace astra {

// ---------------------------------------------------------------------------------------------
// Storage types: two packed elements per 32-bit word, low half at the lower address.
// ---------------------------------------------------------------------------------------------
template <int DT> struct Storage;

template <> struct Storage<ASTRA_BF16> {
    static constexpr int UNITS = 1;  // 16-bit units per element
    static __device__ __forceinline__ void widen2(uint32_t w, float &lo, float &hi) {
        lo = __uint_as_float(w << 16);
        hi = __uint_as_float(w & 0xffff0000u);
    }
    static __device__ __forceinline__ uint32_t narrow2(float lo, float hi) {
        __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);  // one cvt.rn.bf16x2.f32
        return *reinterpret_cast<uint32_t *>(&p);
    }
    static __device__ __forceinline__ float widen1(uint16_t h) {
        return __uint_as_float(static_cast<uint32_t>(h) << 16);
    }
    static __device__ __forceinline__ uint16_t narrow1(float f) {
        return __bfloat16_as_ushort(__float2bfloat16_rn(f));
    }
};

template <> struct Storage<ASTRA_FP16> {
    static constexpr int UNITS = 1;
    static __device__ __forceinline__ void widen2(uint32_t w, float &lo, float &hi) {
        float2 f = __half22float2(*reinterpret_cast<__half2 *>(&w));
        lo = f.x;
        hi = f.y;
    }
    static __device__ __forceinline__ uint32_t narrow2(float lo, float hi) {
        __half2 p = __floats2half2_rn(lo, hi);  // one cvt.rn.f16x2.f32
        return *reinterpret_cast<uint32_t *>(&p);
    }
    static __device__ __forceinline__ float widen1(uint16_t h) {
        return __half2float(__ushort_as_half(h));
    }
    static __device__ __forceinline__ uint16_t narrow1(float f) {
        return __half_as_ushort(__float2half_rn(f));
    }
};

// binary32 storage: an element is two 16-bit units (one 32-bit word) and needs no conversion.
template <> struct Storage<ASTRA_FP32> {
    static constexpr int UNITS = 2;
};

// ---------------------------------------------------------------------------------------------
// A group of N consecutive 16-bit units moved with one global access of 2*N bytes (all tensors are
// addressed in 16-bit units; an element of storage type DT is Storage<DT>::UNITS of them).
// N = 1 is the scalar fallback for odd widths or 2-byte-aligned pointers of the 16-bit types.
// ---------------------------------------------------------------------------------------------
enum class Ld { Stream, StreamReadOnly, Keep };  // once-touched / once-touched and never written / reused (weights)
enum class St { Stream, First, Default };  // a result / one that is read again only much later / kept like anything else

template <int VEC> struct Pack {
    static_assert(VEC == 2 || VEC == 4 || VEC == 8 || VEC == 16, "unsupported vector width");
    static constexpr int WORDS = VEC / 2, UNITS_PER_PACK = VEC;
    uint32_t w[WORDS];
};
template <> struct Pack<1> {
    static constexpr int WORDS = 1, UNITS_PER_PACK = 1;
    uint32_t w[1];  // low 16 bits hold the element
};

template <int VEC, Ld HINT> __device__ __forceinline__ Pack<VEC> load(const uint16_t *p) {
    Pack<VEC> v;
    if constexpr (VEC == 1) {
        uint16_t h;
        if constexpr (HINT == Ld::Keep)
            asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(h) : "l"(p));
        else if constexpr (HINT == Ld::StreamReadOnly)
            asm volatile("ld.global.nc.L1::no_allocate.u16 %0, [%1];" : "=h"(h) : "l"(p));
        else
            asm volatile("ld.global.L1::no_allocate.u16 %0, [%1];" : "=h"(h) : "l"(p) : "memory");
        v.w[0] = h;
    } else if constexpr (VEC == 2) {
        if constexpr (HINT == Ld::Keep)
            asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v.w[0]) : "l"(p));
        else if constexpr (HINT == Ld::StreamReadOnly)
            asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v.w[0]) : "l"(p));
        else
            asm volatile("ld.global.L1::no_allocate.u32 %0, [%1];" : "=r"(v.w[0]) : "l"(p) : "memory");
    } else if constexpr (VEC == 4) {
        if constexpr (HINT == Ld::Keep)
            asm volatile("ld.global.nc.v2.u32 {%0,%1}, [%2];" : "=r"(v.w[0]), "=r"(v.w[1]) : "l"(p));
        else if constexpr (HINT == Ld::StreamReadOnly)
            asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.w[0]), "=r"(v.w[1]) : "l"(p));
        else
            asm volatile("ld.global.L1::no_allocate.v2.u32 {%0,%1}, [%2];"
                         : "=r"(v.w[0]), "=r"(v.w[1]) : "l"(p) : "memory");
    } else if constexpr (VEC == 8) {
        if constexpr (HINT == Ld::Keep)
            asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]) : "l"(p));
        else if constexpr (HINT == Ld::StreamReadOnly)
            asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]) : "l"(p));
        else
            asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]) : "l"(p) : "memory");
    } else {  // 32-byte access (sm_100+)
        if constexpr (HINT == Ld::Keep)
            asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]),
                           "=r"(v.w[4]), "=r"(v.w[5]), "=r"(v.w[6]), "=r"(v.w[7]) : "l"(p));
        else if constexpr (HINT == Ld::StreamReadOnly)
            asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]),
                           "=r"(v.w[4]), "=r"(v.w[5]), "=r"(v.w[6]), "=r"(v.w[7]) : "l"(p));
        else
            asm volatile("ld.global.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]),
                           "=r"(v.w[4]), "=r"(v.w[5]), "=r"(v.w[6]), "=r"(v.w[7]) : "l"(p) : "memory");
    }
    return v;
}

// St::First: the first to leave L2, which then keeps what is read sooner; for the residual of a norm, whose next reader
// comes a layer's matrix products later.  32-byte stores have to ask for it by name, `.cs` does nothing for them.
// What the next operation reads (normalised rows and merged values below kResultsBeyondL2Bytes, activations, all
// destinations of the all-reduce forms) does not get it: the hint then costs more than it gives.  us a call, bf16, with 32-byte stores `.cs` / all of
// them evict-first / the residual's alone.  A norm whose rows are copied in and read back afterwards, then 96 MB
// of other traffic: 30.4 / 30.7 / 30.5 at [1024, 4096], 39.5 / 40.1 / 39.6 at [1024, 8192], 53.4 / 54.3 / 53.4 at [4096,
// 4096], 102.5 / 98.2 / 98.6 at [8192, 4096], 340.3 / 340.7 / 341.4 at [16384, 8192]; without that traffic, so that the
// residual is soon read as well: 19.0 / 20.2 / 19.7 at [1024, 8192], 34.1 / 34.9 / 33.4 at [4096, 4096], 84.9 / 80.5 / 80.9 at
// [8192, 4096].  Norms alone on three sets of operands in turn: 10.3 / 9.6 / 8.5 at [1024, 8192], 9.9 / 9.1 / 7.9 at [2048,
// 4096]; L2-cold 11.2 / 11.2 / 11.0, 11.1 / 11.1 / 10.8, 155.4 / 155.5 / 156.2 at [16384, 8192].  `.cs` / evict-first with
// a reader: merge 18.8 / 19.2 at [1536, 32, 128], 44.7 / 46.0 at [4096, 32, 128]; all-reduce 32.5 / 32.8 at [1024, 4096] of
// 4, 38.8 / 41.3 at [394, 2048] of 8 to 8 destinations, 47.9 / 49.7 at [1024, 4096] of 4 to 4; that reader left out,
// merge 6.53 / 5.92 at [1536, 32, 128] and all-reduce 7.73 / 6.30 at [394, 2048] of 8 to 8.
template <int VEC, St HINT> __device__ __forceinline__ void store(uint16_t *p, const Pack<VEC> &v) {
    if constexpr (VEC == 1) {
        uint16_t h = static_cast<uint16_t>(v.w[0]);
        if constexpr (HINT != St::Default)
            asm volatile("st.global.cs.u16 [%0], %1;" ::"l"(p), "h"(h) : "memory");
        else
            asm volatile("st.global.u16 [%0], %1;" ::"l"(p), "h"(h) : "memory");
    } else if constexpr (VEC == 2) {
        if constexpr (HINT != St::Default)
            asm volatile("st.global.cs.u32 [%0], %1;" ::"l"(p), "r"(v.w[0]) : "memory");
        else
            asm volatile("st.global.u32 [%0], %1;" ::"l"(p), "r"(v.w[0]) : "memory");
    } else if constexpr (VEC == 4) {
        if constexpr (HINT != St::Default)
            asm volatile("st.global.cs.v2.u32 [%0], {%1,%2};" ::"l"(p), "r"(v.w[0]), "r"(v.w[1]) : "memory");
        else
            asm volatile("st.global.v2.u32 [%0], {%1,%2};" ::"l"(p), "r"(v.w[0]), "r"(v.w[1]) : "memory");
    } else if constexpr (VEC == 8) {
        if constexpr (HINT != St::Default)
            asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};"
                         ::"l"(p), "r"(v.w[0]), "r"(v.w[1]), "r"(v.w[2]), "r"(v.w[3]) : "memory");
        else
            asm volatile("st.global.v4.u32 [%0], {%1,%2,%3,%4};"
                         ::"l"(p), "r"(v.w[0]), "r"(v.w[1]), "r"(v.w[2]), "r"(v.w[3]) : "memory");
    } else {  // 32-byte access (sm_100+)
        if constexpr (HINT == St::First)
            asm volatile("st.global.L2::evict_first.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                         ::"l"(p), "r"(v.w[0]), "r"(v.w[1]), "r"(v.w[2]), "r"(v.w[3]),
                           "r"(v.w[4]), "r"(v.w[5]), "r"(v.w[6]), "r"(v.w[7]) : "memory");
        else if constexpr (HINT == St::Stream)
            asm volatile("st.global.cs.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                         ::"l"(p), "r"(v.w[0]), "r"(v.w[1]), "r"(v.w[2]), "r"(v.w[3]),
                           "r"(v.w[4]), "r"(v.w[5]), "r"(v.w[6]), "r"(v.w[7]) : "memory");
        else
            asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                         ::"l"(p), "r"(v.w[0]), "r"(v.w[1]), "r"(v.w[2]), "r"(v.w[3]),
                           "r"(v.w[4]), "r"(v.w[5]), "r"(v.w[6]), "r"(v.w[7]) : "memory");
    }
}

// Pack of VEC elements of storage type DT  <->  VEC floats.
template <int DT, int VEC>
__device__ __forceinline__ void widen(const Pack<VEC * Storage<DT>::UNITS> &v, float (&f)[VEC]) {
    if constexpr (DT == ASTRA_FP32) {
#pragma unroll
        for (int i = 0; i < VEC; ++i) f[i] = __uint_as_float(v.w[i]);
    } else if constexpr (VEC == 1) {
        f[0] = Storage<DT>::widen1(static_cast<uint16_t>(v.w[0]));
    } else {
#pragma unroll
        for (int i = 0; i < VEC / 2; ++i) Storage<DT>::widen2(v.w[i], f[2 * i], f[2 * i + 1]);
    }
}

template <int DT, int VEC>
__device__ __forceinline__ Pack<VEC * Storage<DT>::UNITS> narrow(const float (&f)[VEC]) {
    Pack<VEC * Storage<DT>::UNITS> v;
    if constexpr (DT == ASTRA_FP32) {
#pragma unroll
        for (int i = 0; i < VEC; ++i) v.w[i] = __float_as_uint(f[i]);
    } else if constexpr (VEC == 1) {
        v.w[0] = Storage<DT>::narrow1(f[0]);
    } else {
#pragma unroll
        for (int i = 0; i < VEC / 2; ++i) v.w[i] = Storage<DT>::narrow2(f[2 * i], f[2 * i + 1]);
    }
    return v;
}

// ---------------------------------------------------------------------------------------------
// Rows that start at any element (odd widths, odd pitches): a row is cut into granules of UV units that
// are aligned to 2*UV bytes, so that all but its first and last one are ordinary vector accesses.
// ---------------------------------------------------------------------------------------------
// Units by which p lies beyond the last address that is aligned to UV units.
template <int UV> __host__ __device__ __forceinline__ int misalignment(const uint16_t *p) {
    return static_cast<int>((reinterpret_cast<uint64_t>(p) >> 1) & (UV - 1));
}

// Units [SHIFT, SHIFT + UV) of the 2*UV units lo, hi.  The shift is a constant: an odd one costs one
// funnel shift per word, an even one nothing.  (Selecting among run-time shifts costs 11 selects more per
// 16-byte granule; the callers' shift is the same for a whole block, so they branch over its values once.)
template <int SHIFT, int UV> __device__ __forceinline__ Pack<UV> realign(const Pack<UV> &lo, const Pack<UV> &hi) {
    constexpr int N = UV / 2;
    uint32_t w[2 * N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        w[i] = lo.w[i];
        w[N + i] = hi.w[i];
    }
    Pack<UV> v;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if constexpr (SHIFT % 2 != 0) v.w[i] = __funnelshift_r(w[i + SHIFT / 2], w[i + SHIFT / 2 + 1], 16);
        else v.w[i] = w[i + SHIFT / 2];
    }
    return v;
}

// Runs CALL with the compile-time constant SHIFT set to `shift` (0 <= shift < UV, UV of 8 or 16 in scope,
// shift a multiple of STEP).
#define ASTRA_SHIFT_CASE(K, STEP, CALL)                    \
    case K:                                               \
        if constexpr (K < UV && K % (STEP) == 0) {        \
            constexpr int SHIFT = K;                      \
            CALL;                                         \
        }                                                 \
        break;
#define ASTRA_FOR_SHIFT(shift, STEP, CALL)                                                                        \
    switch (shift) {                                                                                              \
        ASTRA_SHIFT_CASE(0, STEP, CALL) ASTRA_SHIFT_CASE(1, STEP, CALL) ASTRA_SHIFT_CASE(2, STEP, CALL)            \
        ASTRA_SHIFT_CASE(3, STEP, CALL) ASTRA_SHIFT_CASE(4, STEP, CALL) ASTRA_SHIFT_CASE(5, STEP, CALL)            \
        ASTRA_SHIFT_CASE(6, STEP, CALL) ASTRA_SHIFT_CASE(7, STEP, CALL) ASTRA_SHIFT_CASE(8, STEP, CALL)            \
        ASTRA_SHIFT_CASE(9, STEP, CALL) ASTRA_SHIFT_CASE(10, STEP, CALL) ASTRA_SHIFT_CASE(11, STEP, CALL)          \
        ASTRA_SHIFT_CASE(12, STEP, CALL) ASTRA_SHIFT_CASE(13, STEP, CALL) ASTRA_SHIFT_CASE(14, STEP, CALL)         \
        ASTRA_SHIFT_CASE(15, STEP, CALL)                                                                          \
        default: break;                                                                                           \
    }

// The UV units of a row at offset `at` (in units; the row has `width` of them and starts at `row`), unit
// by unit and only those that exist; zeros elsewhere.
template <int UNITS, int UV, Ld HINT>
__device__ __forceinline__ Pack<UV> load_edge(const uint16_t *row, int at, int width) {
    Pack<UV> v;
#pragma unroll
    for (int i = 0; i < UV / 2; ++i) v.w[i] = 0;
#pragma unroll
    for (int k = 0; k < UV; k += UNITS) {
        if (at + k >= 0 && at + k < width) {
            const Pack<UNITS> e = load<UNITS, HINT>(row + at + k);
            if constexpr (UNITS == 2) v.w[k / 2] = e.w[0];
            else v.w[k / 2] |= (k & 1) ? e.w[0] << 16 : (e.w[0] & 0xffffu);
        }
    }
    return v;
}

template <int UNITS, int UV, St HINT>
__device__ __forceinline__ void store_edge(uint16_t *row, int at, int width, const Pack<UV> &v) {
#pragma unroll
    for (int k = 0; k < UV; k += UNITS) {
        if (at + k >= 0 && at + k < width) {
            Pack<UNITS> e;
            e.w[0] = UNITS == 2 ? v.w[k / 2] : ((k & 1) ? v.w[k / 2] >> 16 : v.w[k / 2]);
            store<UNITS, HINT>(row + at + k, e);
        }
    }
}

// Bytes that bring a kernel's parameters to a size that is quick to launch (see launch.cuh); never read.
template <int BYTES> struct LaunchPad {
    uint32_t w[BYTES / 4];
};

// ---------------------------------------------------------------------------------------------
// Programmatic dependent launch.  A kernel launched with the programmatic-stream-serialization
// attribute may be scheduled while the previous kernel in the stream is still draining.  It must
// not touch global memory before `grid_dependency_wait()` returns (the previous grid has then
// completed and its writes are visible), so stream order is preserved; what overlaps is only the
// launch latency and the block prologue.  `grid_launch_dependents()` lets the next kernel in the
// stream do the same with respect to this one.  Both are no-ops for an ordinary launch.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---------------------------------------------------------------------------------------------
// L2 prefetch of a contiguous byte range with one instruction (the bulk-copy engine's prefetch form;
// fire and forget: nothing is returned, nothing has to be waited for).  It needs a 16-byte aligned
// start and a multiple of 16 bytes, so the range is trimmed inward to that; the trimmed edges are
// simply fetched by the loads later.
//
// Use: a block issues it for its inputs BEFORE `grid_dependency_wait()`.  A prefetch consumes no
// data, and L2 is the point of coherence for everything the previous kernel writes, so this is safe
// whatever that kernel does to the same addresses.  What it buys: the request reaches the memory
// system as one contiguous piece before the block's warps have even been through the wait, so the
// first-byte latency overlaps the previous kernel's drain and the block's own prologue.  Measured
// with inputs that are cold in L2: merge 5 % at [8192, 32, 128] and 17 % at [512, 32, 128], silu 5 %
// at [1024, 14336] and 24 % at [128, 14336], rmsnorm 3 % at [1024, 4096]; more when part of the
// input is still in L2.  Only for memory of this GPU.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void prefetch_l2_range(const void *begin, int64_t bytes) {
    const uint64_t lo = (reinterpret_cast<uint64_t>(begin) + 15u) & ~static_cast<uint64_t>(15);
    const uint64_t hi = (reinterpret_cast<uint64_t>(begin) + static_cast<uint64_t>(bytes)) & ~static_cast<uint64_t>(15);
    if (hi > lo) {
        const uint32_t n = static_cast<uint32_t>(hi - lo);
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"(n) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------
// Division of a 31-bit index by a launch-constant divisor: q = (n * mul) >> shift, exact for
// 0 <= n < 2^31 and 1 <= d < 2^31 with shift = 31 + ceil(log2 d), mul = ceil(2^shift / d) <= 2^32 - 1
// (d = 1 is special-cased so that mul fits 32 bits).
// ---------------------------------------------------------------------------------------------
struct FastDiv {
    uint32_t d;
    uint32_t mul;
    uint32_t shift;
    static inline FastDiv make(uint32_t divisor) {
        FastDiv f;
        f.d = divisor;
        uint32_t s = 0;
        while ((1ull << s) < divisor) ++s;
        f.shift = 31 + s;
        uint64_t p = 1ull << f.shift;
        f.mul = static_cast<uint32_t>((p + divisor - 1) / divisor);  // d=1: 2^31; d>=2: < 2^32
        return f;
    }
    __host__ __device__ __forceinline__ uint32_t div(uint32_t n) const {
        return static_cast<uint32_t>((static_cast<uint64_t>(n) * mul) >> shift);
    }
};

}  // namespace astra
