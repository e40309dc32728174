// fused_add_rmsnorm (Astra paper, Table 1, Kernel 2):
//     s = x + r;   r_out <- s;   y <- s / sqrt(mean(s^2) + eps) * w        per row of H elements
// (in place when y is x and r_out is r).
//
// HBM-bound: 8 bytes move per element (x and r read once, y and the new r written once).  One
// thread block owns one row.  In the register-resident kernel each thread keeps its share of the
// binary32 sums s in registers across the row reduction, so the row makes a single trip through
// HBM.  The reduction is the one the paper's optimised kernel uses: shuffles inside each warp, one
// shared-memory slot per warp, then a short combine.  All loads of x and r of a row are issued
// before anything is consumed; the weight (an L2 hit) is fetched while the reduction completes.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "vec.cuh"

namespace astra {

constexpr int kMaxWarps = 32;

// Row-addressed operands.  Pointers and pitches are in 16-bit units.  y may be exactly x and r_out exactly r (the
// in-place form); each thread reads the vectors it later overwrites, so that aliasing is safe.
struct RmsnormOperands {
    const uint16_t *x;
    const uint16_t *r;
    uint16_t *y;
    uint16_t *r_out;
    int64_t x_pitch, r_pitch, y_pitch, r_out_pitch;
};

// Sum over the block; every thread receives the total.  `slots` holds kMaxWarps floats, 16-byte aligned.
// SHORT (at most eight warps): the second stage is two broadcast reads and a tree of additions in every
// thread, whose latency is below that of five more shuffles (1.44 -> 1.34 us at [16, 4096]); in kernels that
// stream it is level.
template <bool SHORT = false> __device__ __forceinline__ float block_sum(float v, float *slots) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nwarps = (blockDim.x + 31) >> 5;
    if (nwarps == 1) return v;
    if (lane == 0) slots[warp] = v;
    __syncthreads();
    float t;
    if constexpr (SHORT) {
        const float4 p = reinterpret_cast<const float4 *>(slots)[0];
        t = (p.x + p.y) + ((nwarps > 2 ? p.z : 0.f) + (nwarps > 3 ? p.w : 0.f));
        if (nwarps > 4) {
            const float4 q = reinterpret_cast<const float4 *>(slots)[1];
            t += (q.x + (nwarps > 5 ? q.y : 0.f)) + ((nwarps > 6 ? q.z : 0.f) + (nwarps > 7 ? q.w : 0.f));
        }
    } else {
        t = lane < nwarps ? slots[lane] : 0.f;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    }
    return t;
}

// s = x + r (one binary32 add per element) and the running sum of squares, two elements per
// instruction with the packed binary32 forms of sm_100 where the vector has an even length (the
// scalar accumulator serves one-element vectors).  Same roundings as the scalar forms.
template <int VEC>
__device__ __forceinline__ void add_and_square(const float (&x)[VEC], const float (&r)[VEC], float (&s)[VEC],
                                               float &acc, float2 &acc2) {
    if constexpr (VEC % 2 == 0) {
#pragma unroll
        for (int k = 0; k < VEC; k += 2) {
            const float2 t = __fadd2_rn(make_float2(x[k], x[k + 1]), make_float2(r[k], r[k + 1]));
            acc2 = __ffma2_rn(t, t, acc2);
            s[k] = t.x;
            s[k + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            s[k] = x[k] + r[k];
            acc = fmaf(s[k], s[k], acc);
        }
    }
}

// y = (s * rstd) * w, packed likewise.
template <int VEC>
__device__ __forceinline__ void scale(const float (&s)[VEC], float rstd, const float (&w)[VEC], float (&y)[VEC]) {
    if constexpr (VEC % 2 == 0) {
        const float2 r2 = make_float2(rstd, rstd);
#pragma unroll
        for (int k = 0; k < VEC; k += 2) {
            const float2 t = __fmul2_rn(__fmul2_rn(make_float2(s[k], s[k + 1]), r2), make_float2(w[k], w[k + 1]));
            y[k] = t.x;
            y[k + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < VEC; ++k) y[k] = s[k] * rstd * w[k];
    }
}

// Largest block the register-resident kernel may be launched with, by vectors per thread: the
// row's binary32 sums plus its packed inputs (counted in 16-bit units per thread) must fit the
// register file.
__host__ __device__ constexpr int rmsnorm_reg_max_threads(int units_per_thread) {
    return units_per_thread <= 16 ? 1024 : (units_per_thread <= 32 ? 512 : 256);
}

// Register-resident row: thread i owns vectors i, i + blockDim.x, ... (at most VPT of them).
// Requires nvec = H / VEC <= VPT * blockDim.x and blockDim.x <= rmsnorm_reg_max_threads(VEC * VPT * UNITS).
// EARLY_W issues the weight loads before the reduction instead of after it (measured: no faster,
// and it costs the registers that decide occupancy).  MINB is the minimum number of resident blocks
// the register allocation must allow; with 16 units per thread in at most four vectors MINB = 2
// caps the kernel at 32 registers, i.e. full occupancy for every block size, which is worth 5 % at
// [16384, 8192] and 27 % at [512, 14336] (896-thread blocks: two per SM instead of one).  The
// four-vector form (8-byte accesses, e.g. H = 4100) fits the cap too; with eight or sixteen narrower
// vectors it would spill, so no cap there.
// DECODE (few rows, at most eight warps): the short second stage of the sum, and the next kernel may start
// when this one's inputs have arrived instead of before they are asked for; its launch then ends just as
// this kernel does, where its blocks would otherwise wait.  Together 1.63 -> 1.39 us at [16, 4096], 1.51 ->
// 1.30 at [16, 2048], 1.87 -> 1.71 at [1, 8192] (device time from a graph).  With more rows the early
// prefetch of the next kernel is worth more (1.9 against 2.2 us at [128, 4096], 11.1 against 11.5 at
// [1024, 8192]), and with more warps neither gains reliably (2.13 against 2.24 us at [16, 11008]).
template <int DT, int VEC, int VPT, Ld LDH = Ld::Stream, St STH = St::Stream, bool EARLY_W = false, bool DECODE = false,
          int MINB = ((VEC * VPT * Storage<DT>::UNITS <= 16 && VPT <= 4 && VEC * Storage<DT>::UNITS >= 4) ? 2 : 1)>
__global__ void __launch_bounds__(rmsnorm_reg_max_threads(VEC * VPT * Storage<DT>::UNITS), MINB)
fused_add_rmsnorm_reg_kernel(RmsnormOperands op, const uint16_t *__restrict__ weight,
                             int H, float eps, float inv_H) {
    constexpr int UV = VEC * Storage<DT>::UNITS;  // 16-bit units per vector
    __shared__ __align__(16) float slots[kMaxWarps];
    const int nvec = H / VEC;
    const int64_t row = blockIdx.x;
    const uint16_t *xr = op.x + row * op.x_pitch;
    const uint16_t *rr = op.r + row * op.r_pitch;
    uint16_t *yr = op.y + row * op.y_pitch;
    uint16_t *ror = op.r_out + row * op.r_out_pitch;
    // the row's two inputs start moving towards L2 while the previous kernel is still draining
    if (threadIdx.x == 0) {
        prefetch_l2_range(xr, static_cast<int64_t>(H) * (2 * Storage<DT>::UNITS));
        prefetch_l2_range(rr, static_cast<int64_t>(H) * (2 * Storage<DT>::UNITS));
    }
    grid_dependency_wait();
    if constexpr (!DECODE) grid_launch_dependents();

    Pack<UV> px[VPT], pr[VPT], pw[VPT];
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < nvec) {
            // x and residual may be rewritten by this same thread below: coherent loads, not .nc
            px[i] = load<UV, LDH>(xr + v * UV);
            pr[i] = load<UV, LDH>(rr + v * UV);
        }
    }
    if constexpr (EARLY_W) {
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const int v = threadIdx.x + i * blockDim.x;
            if (v < nvec) pw[i] = load<UV, Ld::Keep>(weight + v * UV);
        }
    }

    float s[VPT][VEC];
    float acc = 0.f;
    float2 acc2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < nvec) {
            float fx[VEC], fr[VEC];
            widen<DT, VEC>(px[i], fx);
            widen<DT, VEC>(pr[i], fr);
            add_and_square(fx, fr, s[i], acc, acc2);  // the one binary32 add per element
            store<UV, St::First>(ror + v * UV, narrow<DT, VEC>(s[i]));
        }
    }

    if constexpr (!EARLY_W) {
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const int v = threadIdx.x + i * blockDim.x;
            if (v < nvec) pw[i] = load<UV, Ld::Keep>(weight + v * UV);
        }
    }
    if constexpr (DECODE) grid_launch_dependents();
    const float total = block_sum<DECODE>(acc + (acc2.x + acc2.y), slots);
    const float rstd = rsqrtf(fmaf(total, inv_H, eps));

#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < nvec) {
            float fw[VEC], fy[VEC];
            widen<DT, VEC>(pw[i], fw);
            scale(s[i], rstd, fw, fy);
            store<UV, STH>(yr + v * UV, narrow<DT, VEC>(fy));
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Rows that start at any element (odd widths): x, residual and the outputs start at the same place within
// a 32-byte granule, row by row, so the granules that lie inside the row (its body) are 32-byte accesses
// of all four; the few units before and after them (the edge, at most 46) are one element per lane of the
// first two warps.  Only the weight, which starts the same way for every row, lies at an offset to them:
// its two granules per body vector are loaded whole and shifted, by an amount that is the row's.
// ---------------------------------------------------------------------------------------------
struct RaggedRow {
    int first, nvec;  // the body: vectors [first, first + 16 * nvec)
    int shift;        // of the weight against the body
    int edge;         // this thread's edge unit, or -1
};

// The share of thread `thread` of a row of `units` units at `row`.  Body vectors whose weight granules would pass
// the weight's ends are left to the edge: at most 30 units before the body or 30 after it, 46 together.
template <int UNITS>
__host__ __device__ __forceinline__ RaggedRow ragged_row(const uint16_t *row, const uint16_t *weight, int units, int thread) {
    constexpr int UV = 16;
    RaggedRow g;
    g.first = (UV - misalignment<UV>(row)) & (UV - 1);
    g.shift = (misalignment<UV>(weight) + g.first) & (UV - 1);
    if (g.shift > g.first) g.first += UV;
    const int room = units - g.first - (g.shift ? UV - g.shift : 0);
    g.nvec = room > 0 ? room / UV : 0;
    int e = thread * UNITS;
    if (e >= g.first) e += g.nvec * UV;
    g.edge = e < units ? e : -1;
    return g;
}

// The rest of a ragged row once its sums s (and the edge's es) are formed: reduction, weight, y.  EARLY_W
// fetches the weight before the reduction (one vector per thread: no register more than the row's sums
// needed).  STORE(unit offset, pack) writes y.
template <int SHIFT, int DT, int VPT, bool EARLY_W, typename STORE>
__device__ __forceinline__ void ragged_finish(const RaggedRow &g, const uint16_t *weight, float acc, float eps, float inv_H,
                                              float *slots, float (&s)[VPT][16 / Storage<DT>::UNITS], float (&es)[1],
                                              const Pack<Storage<DT>::UNITS> &ew, STORE store_y) {
    constexpr int UV = 16, VEC = UV / Storage<DT>::UNITS;
    Pack<UV> w0[VPT], w1[VPT];
    auto fetch_weight = [&] {
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const int v = threadIdx.x + i * blockDim.x;
            if (v < g.nvec) {
                const uint16_t *w = weight + (g.first + v * UV - SHIFT);
                w0[i] = load<UV, Ld::Keep>(w);
                if constexpr (SHIFT != 0) w1[i] = load<UV, Ld::Keep>(w + UV);
            }
        }
    };
    if constexpr (EARLY_W) fetch_weight();
    const float total = block_sum(acc, slots);
    const float rstd = rsqrtf(fmaf(total, inv_H, eps));
    if constexpr (!EARLY_W) fetch_weight();
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < g.nvec) {
            float fw[VEC], fy[VEC];
            widen<DT, VEC>(realign<SHIFT, UV>(w0[i], w1[i]), fw);
            scale(s[i], rstd, fw, fy);
            store_y(g.first + v * UV, narrow<DT, VEC>(fy));
        }
    }
    if (g.edge >= 0) {
        float fw[1], fy[1];
        widen<DT, 1>(ew, fw);
        scale(es, rstd, fw, fy);
        store_y(g.edge, narrow<DT, 1>(fy));
    }
}

// HBM-bound like the aligned kernel, of which it moves the same bytes in the same widths; what it pays for
// the row's place is the second weight granule, a funnel shift per word of weight and two warps' edge.
// Launched with rmsnorm_ragged_shape's blocks, VPT vectors per thread covering units / 16 of them.
// Measured L2-cold, fp16, against the kernels for 2-, 4- and 8-byte vectors: 41.8 -> 21.3 us at [4096, 4099]
// (19.5 us at 6.9 TB/s), 99.4 -> 28.8 us at [2048, 11007], 142 -> 41.0 us at [2048, 16383], 12.3 -> 6.9 us at
// [1024, 4101], 2.9 -> 2.0 us at [16, 4099], 25.0 -> 21.3 us at [4096, 4098], 79.7 -> 78.8 us at [16384, 4100];
// fp32 56.9 -> 40.9 us at [2048, 8191], 81 -> 43 us at [1024, 16383].  Also tried: 16-byte granules (21.7 and
// 29.2 us at [4096, 4099] and [2048, 11007]), run-time shifts by selects (22.6 and 40.4 us), the edge as
// partial vectors in the main loop (29.8 and 54.6 us: its branches serialise the loads).
// Two vectors per thread hold the sums of 16384 units in two blocks of 512 threads per SM at 64 registers.
constexpr int kRmsnormRaggedMaxThreads = 512, kRmsnormRaggedMinThreads = 64;

// Blocks that an SM holds at once.  Each of its four partitions has 16384 registers, hands them out warp by
// warp in pieces of 256, and a block needs a place for each of its warps: 21 warps of 48 registers fit once, not
// twice, although 2 * 21 * 32 * 48 registers are fewer than 65536 (counting them as two took fp32 [1024, 5152] with
// 2 partials from 17.2 to 20.5 us).
inline int resident_blocks(int regs, int threads) {
    const int warps = (threads + 31) / 32;
    const int by_regs = 4 * (16384 / ((regs * 32 + 255) / 256 * 256)) / warps, by_threads = 64 / warps;
    return by_regs < by_threads ? by_regs : by_threads;
}

// Do T rows of `units` units stay with the other kernels, whose accesses there are of vec = 1, 2, 4 units (8: aligned
// binary32 rows of more than 16384)?  `resident`: blocks of the ragged kernel per SM.
// Odd rows never stay: 19 to 28 against 4 to 7 us at bf16 [400, 8195], 0.6 to 0.8 of the time elsewhere.  4-byte forms only
// where rows are short and about as many as fill the SMs once with the narrow kernel's smaller blocks (1.9 against 2.1
// us at bf16 [400, 1058], where the ragged kernel is at 0.7 to 0.9 of the time from 1800 units on).
// The 8-byte forms move half the instructions of the 4-byte ones and are level or faster (1.9 against 2.1 us at bf16
// [400, 1060], 2.3 and 2.6 at [256, 3164], 3.2 and 3.8 at fp32 [400, 2050]) except where the ragged kernel's one trip is a
// short one (1.90 -> 1.71 us at bf16 [8, 4100]), its wider accesses stream (83.1 -> 81.5 us at [16384, 4100], 4.8 -> 4.1 at
// [600, 4100]), or the rows fit the SMs in one wave of one kernel and not of the other (4.6 -> 4.2 us at bf16 [450, 8196],
// 5.0 against 5.6 at [1500, 2084]).
// Rows of more than 16384 units are otherwise clusters' or swept twice: 7.4 -> 3.7 us at bf16 [128, 16388], 51.6 -> 42.8 at
// fp32 [1024, 16384], 35.6 -> 31.4 at [1024, 11008], 7.1 -> 6.5 at [128, 16384]; but clusters spread a row over several SMs and
// are ahead while rows are few (3.1 against 4.9 us at fp32 [16, 16382], 4.9 and 5.1 at 64 rows, 9.5 and 6.5 at 128; 2.6
// and 3.0 at bf16 [8, 16388]), and where one block fills an SM and a few rows start a second wave (6.1 against 6.8 us at
// fp32 [149 ... 170, 11008]).
inline bool rmsnorm_keeps_narrow(int64_t T, int64_t units, bool binary32, int vec, int resident) {
    const int64_t rows_per_sm = (T + 147) / 148;
    if (vec == 1) return false;
    if (vec == 2) return units < 1536 && T >= 192 && T <= 560;
    if (vec == 8 || units > 16400) return T <= 64 || (units > 18432 && units <= 26624 && T > 148 && T <= 176);
    if (units > 16384) return T <= 32;
    if (units < 2048) return true;
    if (T <= 112) return binary32 ? T > 8 || units > 4608 : T * units > 270000 || units > 6144;
    const int64_t narrow_resident = 64 / ((units + 511) / 512);  // 16 units per thread, every warp slot
    if (T > 256 && rows_per_sm > narrow_resident && rows_per_sm <= resident) return false;
    if (T > 256 && rows_per_sm <= narrow_resident && rows_per_sm > resident) return true;
    if (T <= 512) return T <= 384 || units <= 4608 || units > 6144;
    return (units < 2560 && T < 800) || (units > 6144 && units <= 10240);
}

// Vectors per thread and block size for T rows of `units` units; vpt = 0 where the ragged kernel does not
// apply.  A block has at least 64 threads, one per unit of the longest edge, also where fewer could hold the body.
// One vector per thread up to 320 threads, then two (up to 512 threads), then, for binary32 rows only (half
// the sums per unit), four: 21.3 us with one and 21.6 with two at [4096, 4099], 45.1 and 41.4 us at [4096, 8188],
// 39.2 and 28.8 us at [2048, 11007].  Two also where that makes one wave of what would be a little more (5
// blocks of 256 threads per SM at 48 registers against 8 of 128 at 64: 6.8 -> 6.6 us at [1024, 4101]).
struct RaggedShape {
    int vpt, threads;
};
inline RaggedShape rmsnorm_ragged_shape(int64_t T, int64_t units, bool binary32, int vec) {
    const int64_t nvec = units / 16;
    if (nvec > (binary32 ? 4 : 2) * kRmsnormRaggedMaxThreads) return {0, 0};
    auto threads_for = [&](int v) {
        const int t = ((static_cast<int>(nvec) + v - 1) / v + 31) / 32 * 32;
        return t < kRmsnormRaggedMinThreads ? kRmsnormRaggedMinThreads : t;
    };
    const int64_t wave1 = 148 * (65536 / (48 * threads_for(1))), wave2 = 148 * (65536 / (64 * threads_for(2)));
    RaggedShape sh = {4, threads_for(4)};
    if (nvec <= 320 && !(T > wave1 && T <= wave2)) sh = {1, threads_for(1)};
    else if (nvec <= 2 * kRmsnormRaggedMaxThreads) sh = {2, threads_for(2)};
    const int regs = sh.vpt == 1 ? (binary32 ? 40 : 48) : sh.vpt == 2 ? (binary32 ? 56 : 64) : 96;
    if (rmsnorm_keeps_narrow(T, units, binary32, vec, resident_blocks(regs, sh.threads))) return {0, 0};
    return sh;
}

template <int DT, int VPT, bool EARLY_W, St STH = St::Stream>
__global__ void __launch_bounds__(kRmsnormRaggedMaxThreads, VPT <= 2 ? 2 : 1)
fused_add_rmsnorm_ragged_kernel(RmsnormOperands op, const uint16_t *__restrict__ weight, int H, float eps, float inv_H) {
    constexpr int UV = 16, UNITS = Storage<DT>::UNITS, VEC = UV / UNITS;
    __shared__ __align__(16) float slots[kMaxWarps];
    const int units = H * UNITS;
    const int64_t row = blockIdx.x;
    const uint16_t *xr = op.x + row * op.x_pitch;
    const uint16_t *rr = op.r + row * op.r_pitch;
    uint16_t *yr = op.y + row * op.y_pitch;
    uint16_t *ror = op.r_out + row * op.r_out_pitch;
    if (threadIdx.x == 0) {
        prefetch_l2_range(xr, static_cast<int64_t>(units) * 2);
        prefetch_l2_range(rr, static_cast<int64_t>(units) * 2);
    }
    const RaggedRow g = ragged_row<UNITS>(xr, weight, units, static_cast<int>(threadIdx.x));
    grid_dependency_wait();
    grid_launch_dependents();

    Pack<UV> px[VPT], pr[VPT];
    Pack<UNITS> ex, er, ew;
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < g.nvec) {
            px[i] = load<UV, Ld::Stream>(xr + (g.first + v * UV));
            pr[i] = load<UV, Ld::Stream>(rr + (g.first + v * UV));
        }
    }
    if (g.edge >= 0) {
        ex = load<UNITS, Ld::Stream>(xr + g.edge);
        er = load<UNITS, Ld::Stream>(rr + g.edge);
        ew = load<UNITS, Ld::Keep>(weight + g.edge);
    }
    float s[VPT][VEC], es[1];
    float acc = 0.f;
    float2 acc2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < g.nvec) {
            float fx[VEC], fr[VEC];
            widen<DT, VEC>(px[i], fx);
            widen<DT, VEC>(pr[i], fr);
            add_and_square(fx, fr, s[i], acc, acc2);
            store<UV, St::First>(ror + (g.first + v * UV), narrow<DT, VEC>(s[i]));
        }
    }
    if (g.edge >= 0) {
        float fx[1], fr[1];
        widen<DT, 1>(ex, fx);
        widen<DT, 1>(er, fr);
        add_and_square(fx, fr, es, acc, acc2);
        store<UNITS, St::First>(ror + g.edge, narrow<DT, 1>(es));
    }
    auto store_y = [&](int at, const auto &v) { store<std::decay_t<decltype(v)>::UNITS_PER_PACK, STH>(yr + at, v); };
    ASTRA_FOR_SHIFT(g.shift, UNITS,
                    (ragged_finish<SHIFT, DT, VPT, EARLY_W>(g, weight, acc + (acc2.x + acc2.y), eps, inv_H, slots, s, es, ew,
                                                            store_y)))
}

// Rows too wide for one block's registers: a thread-block cluster owns the row.  Each block keeps
// its contiguous share of the row in registers exactly as above and reduces it; the per-block
// partial sums are then exchanged through distributed shared memory (every block reads every
// partial, in rank order, so all blocks form the same total bit for bit), and each block finishes
// its share.  The row still makes one trip through HBM.  The two cluster barriers are hardware
// barriers that every thread of every block reaches unconditionally (blocks without work included):
// the first publishes the partials; the second, split into an arrive right after the partials are
// read and a wait at the very end, keeps each block's shared memory alive until all its peers have
// read it without stalling the final stores.
// (scalar arithmetic here: the packed forms cost the registers that keep this kernel at full
// occupancy, which matters more: 5.4 against 4.5 TB/s at [2048, 14336] fp32)
template <int DT, int VEC, int VPT, int MINB = ((VEC * VPT * Storage<DT>::UNITS <= 16 && VPT <= 2) ? 2 : 1)>
__global__ void __launch_bounds__(rmsnorm_reg_max_threads(VEC * VPT * Storage<DT>::UNITS), MINB)
fused_add_rmsnorm_cluster_kernel(RmsnormOperands op, const uint16_t *__restrict__ weight,
                                 int H, float eps, float inv_H) {
    namespace cg = cooperative_groups;
    constexpr int UV = VEC * Storage<DT>::UNITS;
    __shared__ __align__(16) float slots[kMaxWarps];
    __shared__ float block_partial;
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned nblocks = cluster.num_blocks();
    const unsigned rank = cluster.block_rank();
    const int nvec = H / VEC;
    const int chunk = (nvec + nblocks - 1) / nblocks;  // vectors per block (the last may hold fewer)
    const int first = rank * chunk;
    const int count = max(0, min(chunk, nvec - first));
    const int64_t row = blockIdx.x / nblocks;
    const uint16_t *xr = op.x + row * op.x_pitch + static_cast<int64_t>(first) * UV;
    const uint16_t *rr = op.r + row * op.r_pitch + static_cast<int64_t>(first) * UV;
    uint16_t *yr = op.y + row * op.y_pitch + static_cast<int64_t>(first) * UV;
    uint16_t *ror = op.r_out + row * op.r_out_pitch + static_cast<int64_t>(first) * UV;
    const uint16_t *wr = weight + static_cast<int64_t>(first) * UV;
    if (threadIdx.x == 0) {
        prefetch_l2_range(xr, static_cast<int64_t>(count) * UV * 2);
        prefetch_l2_range(rr, static_cast<int64_t>(count) * UV * 2);
    }
    grid_dependency_wait();
    grid_launch_dependents();

    Pack<UV> px[VPT], pr[VPT], pw[VPT];
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < count) {
            px[i] = load<UV, Ld::Stream>(xr + v * UV);
            pr[i] = load<UV, Ld::Stream>(rr + v * UV);
        }
    }
    float s[VPT][VEC];
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < count) {
            float fx[VEC], fr[VEC];
            widen<DT, VEC>(px[i], fx);
            widen<DT, VEC>(pr[i], fr);
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                s[i][k] = fx[k] + fr[k];
                acc = fmaf(s[i][k], s[i][k], acc);
            }
            store<UV, St::First>(ror + v * UV, narrow<DT, VEC>(s[i]));
        }
    }
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < count) pw[i] = load<UV, Ld::Keep>(wr + v * UV);
    }
    const float mine = block_sum(acc, slots);
    if (threadIdx.x == 0) block_partial = mine;
    cluster.sync();
    float total = 0.f;
    for (unsigned b = 0; b < nblocks; ++b) total += *cluster.map_shared_rank(&block_partial, b);
    cluster.barrier_arrive();  // "I have read my peers' partials"; waited for just before exit
    const float rstd = rsqrtf(fmaf(total, inv_H, eps));
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < count) {
            float fw[VEC], fy[VEC];
            widen<DT, VEC>(pw[i], fw);
#pragma unroll
            for (int k = 0; k < VEC; ++k) fy[k] = s[i][k] * rstd * fw[k];
            store<UV, St::Stream>(yr + v * UV, narrow<DT, VEC>(fy));
        }
    }
    cluster.barrier_wait();  // no block leaves while a peer may still read its shared memory
}

// Any H: two sweeps over the row.  The first only reads (x, r) and accumulates the sum of squares;
// the second re-reads them (the row was just touched, so it comes from L2), recomputes the same
// binary32 sums, and writes both outputs.  Nothing is written before the norm is known, so the
// in-place update cannot disturb the reduction.
template <int DT, int VEC>
__global__ void fused_add_rmsnorm_twopass_kernel(RmsnormOperands op,
                                                 const uint16_t *__restrict__ weight,
                                                 int H, float eps, float inv_H) {
    constexpr int UV = VEC * Storage<DT>::UNITS;  // 16-bit units per vector
    __shared__ __align__(16) float slots[kMaxWarps];
    const int nvec = H / VEC;
    const int64_t row = blockIdx.x;
    const uint16_t *xr = op.x + row * op.x_pitch;
    const uint16_t *rr = op.r + row * op.r_pitch;
    uint16_t *yr = op.y + row * op.y_pitch;
    uint16_t *ror = op.r_out + row * op.r_out_pitch;
    grid_dependency_wait();
    grid_launch_dependents();

    float acc = 0.f;
    for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
        float fx[VEC], fr[VEC];
        widen<DT, VEC>(load<UV, Ld::Stream>(xr + v * UV), fx);
        widen<DT, VEC>(load<UV, Ld::Stream>(rr + v * UV), fr);
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            const float s = fx[k] + fr[k];
            acc = fmaf(s, s, acc);
        }
    }
    const float total = block_sum(acc, slots);
    const float rstd = rsqrtf(fmaf(total, inv_H, eps));

    for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
        float fx[VEC], fr[VEC], fw[VEC], fs[VEC], fy[VEC];
        widen<DT, VEC>(load<UV, Ld::Stream>(xr + v * UV), fx);
        widen<DT, VEC>(load<UV, Ld::Stream>(rr + v * UV), fr);
        widen<DT, VEC>(load<UV, Ld::Keep>(weight + v * UV), fw);
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            fs[k] = fx[k] + fr[k];
            fy[k] = fs[k] * rstd * fw[k];
        }
        store<UV, St::First>(ror + v * UV, narrow<DT, VEC>(fs));
        store<UV, St::Stream>(yr + v * UV, narrow<DT, VEC>(fy));
    }
}

}  // namespace astra
