// silu_and_mul (Astra paper, Table 1, Kernel 3):  out = a * sigmoid(a) * b,  row = [a | b].
//
// Elementwise and HBM-bound: 6 bytes move per output (4 read, 2 written).  Each thread owns UNROLL
// vectors of VEC elements; all its 2*UNROLL loads are issued before the first use so that enough
// bytes are in flight per SM to cover HBM latency.  The sigmoid costs two special-function ops per
// element (ex2 and rcp, the fast-math forms the paper's optimised kernel also turns to), in
// binary32, with one rounding at the store.  Instruction count matters even though the kernel is
// HBM-bound: under a sustained power cap the SM clock (and with it the on-chip fabric) drops as
// issue activity rises (1.5 to 1.7 GHz at 1 kW), so the arithmetic is kept to the packed two-wide forms and,
// for all but very negative gates, to half the instructions of the overflow-free form.  Sustained, L2-cold, against
// that form for all elements: 101.7 -> 100.2 us at bf16 [8192, 14336], 57.9 -> 55.7 at [4000, 14333], 36.0 -> 34.6 at fp16
// [8192, 4099] (21.8 instead of 25.9 million warp instructions at [4096, 14336]), 34.5 -> 33.0 at [8192, 4100], 15.2 -> 14.8 at [1000, 14337], 13.4 -> 13.1 at [1024, 14336].
#pragma once

#include <type_traits>

#include "vec.cuh"

namespace astra {

// SiLU(a) * b in binary32.  From a = -40 up directly, a / (1 + e^{-a}) * b.  Below, where e^{-a} may overflow, sigmoid(a) =
// e^a (1 + e^a is 1 there), formed as h*h with h = e^{a/2} = 2^{a * log2(e)/2}: h stays a normal number down to a = -174,
// and the (non-flushing) product h*h reaches the subnormals, so a * e^{a} * b is still produced where e^{a} alone is
// below 2^-126; beyond a = -174 the true result is below every representable magnitude anyway.  Against 64 bits,
// binary32: largest relative error 5.9e-7 for |a| < 10 and 2.0e-6 above -40 (6.6e-7 and 2.0e-6 with the overflow-free
// form).  Which form an element takes depends on nothing but itself, so results do not depend on how a row is cut
// into vectors.
constexpr float kLog2e = 1.4426950408889634f, kHalfLog2e = 0.7213475204444817f, kSiluDirect = -40.0f;

__device__ __forceinline__ float silu_mul(float a, float b) {
    const bool far = a < kSiluDirect;
    float e, d;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(a * (far ? kHalfLog2e : -kLog2e)));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(d) : "f"(e + 1.0f));
    return a * (far ? e * e : d) * b;
}

// Two elements, with the packed binary32 instructions of sm_100 (two multiplies or adds per issue slot); the
// two special-function ops per element stay scalar.  Same arithmetic, element by element, as silu_mul; without FAR
// neither may be below -40.
template <bool FAR> __device__ __forceinline__ float2 silu_mul2(float2 a, float2 b) {
    const bool far_x = FAR && a.x < kSiluDirect, far_y = FAR && a.y < kSiluDirect;
    const float2 arg = __fmul2_rn(a, make_float2(far_x ? kHalfLog2e : -kLog2e, far_y ? kHalfLog2e : -kLog2e));
    float2 e, d;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(arg.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(arg.y));
    const float2 den = __fadd2_rn(e, make_float2(1.0f, 1.0f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(d.x) : "f"(den.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(d.y) : "f"(den.y));
    if constexpr (FAR) {
        const float2 t = __fmul2_rn(e, e);
        d = make_float2(far_x ? t.x : d.x, far_y ? t.y : d.y);
    }
    return __fmul2_rn(__fmul2_rn(a, d), b);
}

// Is any element below -40 (or, of the 16-bit types, a NaN with its sign set)?  The patterns of negative numbers grow
// with their magnitude, so 16-bit elements are compared as unsigned integers, two per instruction.
template <int DT, int UV> __device__ __forceinline__ bool any_far(const Pack<UV> &a) {
    constexpr int WORDS = Pack<UV>::WORDS;
    if constexpr (DT == ASTRA_FP32) {
        float least = kSiluDirect;
#pragma unroll
        for (int i = 0; i < WORDS; ++i) least = fminf(least, __uint_as_float(a.w[i]));
        return least < kSiluDirect;
    } else {
        constexpr uint32_t limit = DT == ASTRA_FP16 ? 0xd100d100u : 0xc220c220u;  // -40, twice
        uint32_t most = limit;
#pragma unroll
        for (int i = 0; i < WORDS; i += 2)
            most = i + 1 < WORDS ? __vimax3_u16x2(most, a.w[i], a.w[i + 1]) : __vmaxu2(most, a.w[i]);
        return most != limit;
    }
}

// SiLU(a) * b on whole packs.  A warp in which any element is below -40 takes the form with the selects as a whole, so that
// no lane waits for another's branch.  Vector by vector, in a rolled loop, such gates cost up to twice the time; loop /
// this, us, L2-cold, bf16: 12.85 / 6.78 at [512, 14336] with 1 % of the gates at -60 (6.89 with the overflow-free form
// throughout), 80.6 / 50.3 at [4096, 14336], 9.42 / 6.74 at [512, 14336] with all, 1.56 / 1.45 at [16, 14336] with one
// channel, 47.6 / 32.7 at fp16 [8192, 4099] with 1 %; without such gates 6.67 / 6.66 at [512, 14336].  The operands are
// widened within each branch: ahead of it, 32-byte vectors take 48 registers instead of 32 (6.97 us there).
template <int DT, int UV> __device__ __forceinline__ Pack<UV> silu_mul_pack(const Pack<UV> &a, const Pack<UV> &b) {
    constexpr int VEC = UV / Storage<DT>::UNITS;
    if constexpr (VEC == 1) {
        float fa[VEC], fb[VEC], fo[VEC];
        widen<DT, VEC>(a, fa);
        widen<DT, VEC>(b, fb);
        fo[0] = silu_mul(fa[0], fb[0]);
        return narrow<DT, VEC>(fo);
    } else {
        auto each_pair = [&](auto far) {
            float fa[VEC], fb[VEC], fo[VEC];
            widen<DT, VEC>(a, fa);
            widen<DT, VEC>(b, fb);
#pragma unroll
            for (int i = 0; i < VEC; i += 2) {
                const float2 o = silu_mul2<decltype(far)::value>(make_float2(fa[i], fa[i + 1]), make_float2(fb[i], fb[i + 1]));
                fo[i] = o.x;
                fo[i + 1] = o.y;
            }
            return narrow<DT, VEC>(fo);
        };
        if (__any_sync(__activemask(), any_far<DT, UV>(a))) return each_pair(std::true_type{});
        return each_pair(std::false_type{});
    }
}

// Flat indexing: vector v of the output covers out[row, col*VEC .. col*VEC+VEC) with
// row = v / nvec, col = v % nvec, nvec = D / VEC.  A block handles THREADS*UNROLL consecutive vectors.
// gate and up are addressed separately (pointers and row pitches in 16-bit units), which covers both the packed
// row [a | b] (up = gate + D, equal pitches) and two independent tensors.
template <int DT, int VEC, int UNROLL, int THREADS, Ld LDH = Ld::StreamReadOnly, St STH = St::Stream,
          int PF_VECS = 0>
__global__ void __launch_bounds__(THREADS)
silu_and_mul_kernel(uint16_t *__restrict__ out, const uint16_t *__restrict__ gate,
                    const uint16_t *__restrict__ up, uint32_t total_vecs, FastDiv nvec,
                    int64_t out_pitch, int64_t gate_pitch, int64_t up_pitch, LaunchPad<24>) {
    constexpr int UV = VEC * Storage<DT>::UNITS;  // 16-bit units per vector
    const uint32_t base = blockIdx.x * (THREADS * UNROLL) + threadIdx.x;
    // Ahead of the dependency wait, the block asks for the gate and up bytes of its vectors to be
    // brought into L2: PF_VECS vectors per request (0 = no prefetch), each request cut at a row end.
    if constexpr (PF_VECS > 0) {
        const uint32_t first = blockIdx.x * (THREADS * UNROLL);
        const uint32_t piece = threadIdx.x * PF_VECS;  // thread t asks for vectors [first + piece, + PF_VECS)
        if (piece < THREADS * UNROLL && first + piece < total_vecs) {
            const uint32_t v0 = first + piece;
            const uint32_t row = nvec.div(v0);
            const uint32_t col = v0 - row * nvec.d;
            uint32_t n = min(static_cast<uint32_t>(PF_VECS), total_vecs - v0);
            n = min(n, nvec.d - col);
            const int64_t c = static_cast<int64_t>(col) * UV;
            prefetch_l2_range(gate + (static_cast<int64_t>(row) * gate_pitch + c), static_cast<int64_t>(n) * UV * 2);
            prefetch_l2_range(up + (static_cast<int64_t>(row) * up_pitch + c), static_cast<int64_t>(n) * UV * 2);
        }
    }
    grid_dependency_wait();
    grid_launch_dependents();
    Pack<UV> a[UNROLL], b[UNROLL];
#pragma unroll
    for (int j = 0; j < UNROLL; ++j) {
        const uint32_t v = base + j * THREADS;
        if (v < total_vecs) {
            const uint32_t row = nvec.div(v);
            const uint32_t col = v - row * nvec.d;
            const int64_t c = static_cast<int64_t>(col) * UV;
            a[j] = load<UV, LDH>(gate + (static_cast<int64_t>(row) * gate_pitch + c));
            b[j] = load<UV, LDH>(up + (static_cast<int64_t>(row) * up_pitch + c));
        }
    }
#pragma unroll
    for (int j = 0; j < UNROLL; ++j) {
        const uint32_t v = base + j * THREADS;
        if (v < total_vecs) {
            const uint32_t row = nvec.div(v);
            const uint32_t col = v - row * nvec.d;
            store<UV, STH>(out + (static_cast<int64_t>(row) * out_pitch + static_cast<int64_t>(col) * UV),
                            silu_mul_pack<DT, UV>(a[j], b[j]));
        }
    }
}

// Rows that start at any element: the widths and pitches whose common divisor leaves less than a 16-byte
// access (odd widths above all, where the flat kernel moves one element per load).
//
// The output row is cut into 16-byte granules that are aligned in the OUTPUT; a thread owns one.  Its 8
// units of gate (and of up) straddle two aligned granules of that input, at an offset that is the same
// for the whole row: both are loaded with 16-byte accesses (the second one is the neighbour thread's first,
// an L1 hit) and the 8 units are taken out of them with ASTRA_FOR_SHIFT, uniformly for the block, which
// covers one piece of one row.
//
// What bounds it: HBM, then issue slots (two loads, up to eight shifts and the edges' tests more per granule than the
// aligned kernel).  Measured L2-cold, fp16, against the narrow flat
// kernels: 28.5 -> 14.1 us at [1000, 14337] (12.5 us at 6.9 TB/s), 64.0 -> 33.7 us at [8192, 4099], 39.9 -> 33.7 us at
// [8192, 4098], 5.69 -> 4.5 us at [300, 11010]; fp32 16.0 -> 13.1 us at [1000, 7001].  Also tried: flat
// indexing over all rows' granules (15.3 and 33.8 us: the shifts are then per thread and need selects),
// the neighbour's granule by shuffles (18.6 and 43.9 us), two granules per thread (16.5 us), 32-byte
// granules (16.0 and 37.7 us), blocks of 256 and 448 threads instead of about 192 (14.7 and 15.9 us).
//
// Accesses stay inside mapped memory: a granule of a row other than the launch's first and last may reach up to 14
// units into what lies before it or 15 into what lies after, which silu_ragged_end_rows makes sure of (and the
// launch code that the output shares no address range with the inputs, so that nothing that is written is read);
// the rows it names load the few granules that would pass their ends element by element, and so are the ends of
// every output row stored.
constexpr int kSiluRaggedMaxThreads = 256;
struct RaggedGranule {
    int at;                // first unit of the output granule, in the row (negative before its start)
    int shift_a, shift_b;  // of its units in the aligned granules of gate and up
    bool whole;            // the aligned granules lie inside the tensors
};
__host__ __device__ __forceinline__ RaggedGranule ragged_granule(const uint16_t *out_row, const uint16_t *gate_row,
                                                                 const uint16_t *up_row, int granule, int D, bool end_row) {
    constexpr int UV = 8;
    const int lead = misalignment<UV>(out_row);
    RaggedGranule g;
    g.at = granule * UV - lead;
    g.shift_a = (misalignment<UV>(gate_row) - lead) & (UV - 1);
    g.shift_b = (misalignment<UV>(up_row) - lead) & (UV - 1);
    g.whole = !(end_row && (g.at < UV || g.at + 2 * UV > D));
    return g;
}

// Which rows of less than 16-byte alignment (vec units per access of the flat kernel) come here: not short rows of 4-
// and 8-byte vectors, whose blocks would be too small (11.2 against 17.7 us at [16384, 514]), nor a single row of
// them that is little longer, both of whose ends are loaded by element (1.07 against 1.14 us at [1, 1028]), nor long streams
// of 8-byte vectors of the 16-bit types (30.3 against 31.4 us at [8192, 4100], 50.4 against 53.5 us at [4000, 14332]; level at
// [4000, 4100], 6.0 -> 5.0 us at [1000, 4100], 14.0 -> 13.5 us at [1000, 14332]; fp32, with half the arithmetic per byte, gains
// at every size: 29.7 -> 28.4 us at [4000, 4098]).
#ifndef ASTRA_SILU_RAGGED_MIN_UNITS
#define ASTRA_SILU_RAGGED_MIN_UNITS 1024
#endif
constexpr int64_t kSiluRaggedMinUnits = ASTRA_SILU_RAGGED_MIN_UNITS, kSiluRaggedMaxUnits = 1ll << 24;
constexpr int64_t kSiluRaggedMaxTotal = 1ll << 24;  // units of output, for 8-byte vectors of the 16-bit types
inline bool silu_takes_ragged(int64_t T, int64_t D, bool binary32, int vec) {
    if (vec >= 8 || D > kSiluRaggedMaxUnits) return false;
    if (vec == 1) return D >= kSiluRaggedMinUnits / 2;
    return D >= kSiluRaggedMinUnits && T > (kSiluRaggedMinUnits * (vec == 4 ? 8 : 5) / 4 - 1) / D &&
            !(vec == 4 && !binary32 && T > kSiluRaggedMaxTotal / D);
}

// The rows of a launch of `rows` whose granules must not pass their ends are row 0 and those from the returned one on:
// the last row, or all where the memory between two rows may not exist.  Between two rows less than a page (4096
// bytes) apart there is no page without a part of one of them; gate and up that fill one another's gaps (the
// packed form [gate | up], padded or not) leave only the rest.  Pitches in units.
inline uint32_t silu_ragged_end_rows(uint32_t rows, const uint16_t *gate, const uint16_t *up, int64_t D, int64_t gate_pitch,
                                     int64_t up_pitch) {
    const bool packed = gate_pitch == up_pitch && (up == gate + D || gate == up + D);
    const int64_t taken = packed ? 2 * D : D;
    const int64_t gap = (gate_pitch > up_pitch ? gate_pitch : up_pitch) - taken;
    return gap < 2048 ? rows - 1 : 0;
}

template <int DT, int ALIGN>
__global__ void __launch_bounds__(kSiluRaggedMaxThreads, 8)
silu_and_mul_ragged_kernel(uint16_t *__restrict__ out, const uint16_t *__restrict__ gate,
                           const uint16_t *__restrict__ up, FastDiv pieces, uint32_t end_rows, int D,
                           int64_t out_pitch, int64_t gate_pitch, int64_t up_pitch, LaunchPad<16>) {
    constexpr int UV = 8, UNITS = Storage<DT>::UNITS;
    const uint32_t row = pieces.div(blockIdx.x);
    const int first = static_cast<int>((blockIdx.x - row * pieces.d) * blockDim.x) * UV;
    const uint16_t *a = gate + static_cast<int64_t>(row) * gate_pitch;
    const uint16_t *b = up + static_cast<int64_t>(row) * up_pitch;
    uint16_t *o = out + static_cast<int64_t>(row) * out_pitch;
    if (threadIdx.x == 0) {
        const int64_t n = min(static_cast<int>(blockDim.x) * UV, D - first);
        if (n > 0) {
            prefetch_l2_range(a + first, n * 2);
            prefetch_l2_range(b + first, n * 2);
        }
    }
    const RaggedGranule g = ragged_granule(o, a, b, first / UV + static_cast<int>(threadIdx.x), D,
                                           row == 0 || row >= end_rows);
    grid_dependency_wait();
    grid_launch_dependents();
    if (g.at >= D) return;
    Pack<UV> va, vb;
    if (g.whole) {
        // cached loads: the second granule is some other thread's first
        const uint16_t *pa = a + (g.at - g.shift_a), *pb = b + (g.at - g.shift_b);
        const Pack<UV> a0 = load<UV, Ld::Keep>(pa), b0 = load<UV, Ld::Keep>(pb);
        Pack<UV> a1, b1;
        if (g.shift_a) a1 = load<UV, Ld::Keep>(pa + UV);
        if (g.shift_b) b1 = load<UV, Ld::Keep>(pb + UV);
        ASTRA_FOR_SHIFT(g.shift_a, ALIGN, va = (realign<SHIFT, UV>(a0, a1)))
        ASTRA_FOR_SHIFT(g.shift_b, ALIGN, vb = (realign<SHIFT, UV>(b0, b1)))
    } else {
        va = load_edge<UNITS, UV, Ld::StreamReadOnly>(a, g.at, D);
        vb = load_edge<UNITS, UV, Ld::StreamReadOnly>(b, g.at, D);
    }
    const Pack<UV> v = silu_mul_pack<DT, UV>(va, vb);
    if (g.at >= 0 && g.at + UV <= D) store<UV, St::Stream>(o + g.at, v);
    else store_edge<UNITS, UV, St::Stream>(o, g.at, D, v);
}

}  // namespace astra
