// fused_allreduce_add_rmsnorm: fused_add_rmsnorm (Astra paper, Table 1, Kernel 2) on a hidden state
// that arrives as N partial sums, one per tensor-parallel rank:
//     x = x_0 + x_1 + ... + x_{N-1};   s = x + r;   r_out <- s;   y <- s / sqrt(mean(s^2) + eps) * w
// Every addition is one binary32 addition, in rank order, the residual last, so that all ranks of a
// group that run this on the same partials produce identical bits.
//
// One-shot form: each rank reads all N partials of the rows it normalises (its own from local
// memory, the others through peer-mapped addresses) and writes only its own memory.  Two-shot form
// (for batches large enough that the N-fold read would be bound by the links): each rank does this
// for its own block of rows only and stores the results to every rank's buffers, so each element
// crosses the links once as a partial and once as a result instead of N - 1 times.
// All loads and stores are plain per-thread `ld.global` / `st.global` (no multicast, no bulk or
// tensor-map copies), so a partial or a destination may live in another GPU's memory.  The kernel
// waits for nothing: the caller orders it after every rank has finished writing its partial and
// orders the consumers after it (stream events, a host barrier).
//
// HBM/NVLink-bound: (N + 1 + Dy + Dr) * 2 bytes per element of 16-bit storage (N partials and r read,
// y written to Dy destinations and the new residual to Dr; N + 3 in the one-shot form).  One block owns a row and keeps the running binary32 sums in registers; the
// partials are fetched GROUP at a time so that GROUP (+1 for the residual) vector loads per vector
// position are in flight before the first addition (GROUP = 2 measured best; see the launch code).
#pragma once

#include "fused_add_rmsnorm.cuh"

namespace astra {

constexpr int kMaxParts = 16;

// Dense [T, H] operands (row pitch = H).  Pointers are in 16-bit units.  Each result goes to one or
// more destinations (the same bytes to each): with one destination apiece this is the one-shot
// all-reduce; with one destination per rank it is the two-shot form, in which a rank reduces and
// normalises only its own row block and pushes the results into every rank's buffers.  A residual
// destination may be exactly r (each thread reads the residual vectors it later overwrites); the
// destinations overlap nothing else.
struct AllreduceOperands {
    const uint16_t *part[kMaxParts];  // rank order
    const uint16_t *r;
    uint16_t *y_out[kMaxParts];
    uint16_t *r_out[kMaxParts];
    int n_parts, n_y, n_r;
};

// The same vector to each of the first n destinations, with plain per-thread stores (a destination
// may be another GPU's memory).  Unrolled and left by a break, so every copy has a constant index.
template <int UV>
__device__ __forceinline__ void store_to_all(uint16_t *const (&dst)[kMaxParts], int n, int64_t at, const Pack<UV> &v) {
#pragma unroll
    for (int d = 0; d < kMaxParts; ++d) {
        if (d >= n) break;
        store<UV, St::Stream>(dst[d] + at, v);
    }
}

// s += x, two elements per instruction where the vector length is even (same roundings as scalar adds).
template <int VEC>
__device__ __forceinline__ void accumulate(float (&s)[VEC], const float (&x)[VEC]) {
    if constexpr (VEC % 2 == 0) {
#pragma unroll
        for (int k = 0; k < VEC; k += 2) {
            const float2 t = __fadd2_rn(make_float2(s[k], s[k + 1]), make_float2(x[k], x[k + 1]));
            s[k] = t.x;
            s[k + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < VEC; ++k) s[k] += x[k];
    }
}

// Largest block of the register-resident kernel: a thread holds its share of the row as binary32 sums
// (one register per element) plus GROUP + 1 packed input copies of it, and the register file is
// 64 K registers per block.  `units` = 16-bit units of the row per thread.
// With two loads in flight 16 units per thread need 54 to 56 registers, so even a 1024-thread block
// fits; that matters for rows of more than 8192 units, where one fat block per SM with one vector per
// thread beat two vectors per thread in half as many threads by 3 to 9 % (e.g. 157.9 -> 143.1 us at
// [4096, 16384] with 4 partials, 82.2 -> 77.4 us at [4096, 11008] with 2).
// One load in flight serves binary32 rows of up to 64 units per thread (32 sums).
__host__ __device__ constexpr int allreduce_reg_max_threads(int units, int group) {
    return group == 1 ? 512
         : group > 4 ? (units <= 16 ? 512 : 128)
         : group > 2 ? (units <= 8 ? 1024 : (units <= 16 ? 512 : 256))
                     : (units <= 16 ? 1024 : 512);
}

// Register-resident row: thread i owns vectors i, i + blockDim.x, ... (at most VPT of them).
// Requires nvec = H / VEC <= VPT * blockDim.x and blockDim.x <= allreduce_reg_max_threads(...), or
// blockDim.x <= kAllreduceDenseThreads for the DENSE instantiation: blocks of at most 256 threads
// whose register allocation is held to 48 so that five of them are resident per SM instead of four
// (for two loads in flight and 16 units per thread that costs no spill).  Measured at [8192, 4096],
// L2-cold: 50.8 -> 50.5 us with 2 partials, 71.5 -> 70.4 us with 4, 112.2 -> 110.3 us with 8; at
// [1024, 4096] it is neutral or slower (16.1 -> 16.5 us with 8 partials), so the launch code uses it
// for long streams only.
constexpr int kAllreduceDenseThreads = 256;
constexpr int kAllreduceDenseBlocks = 5;

//
// LATE_R requests the residual after the partials instead of with the first of them, which frees its
// registers while they are summed, and asks for two resident blocks of up to 448 threads: two vectors per thread
// with two partial loads in flight are held to 72 registers instead of 96 (the 16-bit forms spill 52 to 60 bytes for it,
// the ragged fp16 form 4; binary32 needs 59 and 63), and two blocks fit an SM instead of one.  For rows of 10241
// to 14336 units, where every other shape leaves one block per SM that idles at its barrier, L2-cold, with
// 2 / 4 / 8 partials: 79.7 -> 67.9, 112.7 -> 92.2, 171.0 -> 145.3 us at [4096, 11008] (65.4 / 91.5 / 143.8 us at
// 6.9 TB/s) and 93.2 -> 86.1, 133.2 -> 119.4, 203.5 -> 188.2 us at [4096, 14336]; no gain where two blocks fit
// anyway (61.1 against 62.8 us at [4096, 10240]).
constexpr int kAllreduceLateThreads = 448;

template <int DT, int VEC, int VPT, int GROUP, bool DENSE = false, bool LATE_R = false>
__global__ void __launch_bounds__(LATE_R ? kAllreduceLateThreads : DENSE ? kAllreduceDenseThreads
                                                                  : allreduce_reg_max_threads(VEC * VPT * Storage<DT>::UNITS, GROUP),
                                  LATE_R ? 2 : DENSE ? kAllreduceDenseBlocks : 1)
fused_allreduce_add_rmsnorm_reg_kernel(const __grid_constant__ AllreduceOperands op,
                                       const uint16_t *__restrict__ weight, int H, float eps, float inv_H, LaunchPad<40>) {
    constexpr int UV = VEC * Storage<DT>::UNITS;  // 16-bit units per vector
    __shared__ __align__(16) float slots[kMaxWarps];
    const int nvec = H / VEC;
    const int64_t row = static_cast<int64_t>(blockIdx.x) * H * Storage<DT>::UNITS;  // first unit of the row
    const int n = op.n_parts;
    // The residual row is this GPU's own memory: ask for it ahead of the dependency wait.  The partials
    // may be another GPU's memory and are left to the ordinary loads below.
    if (threadIdx.x == 0) prefetch_l2_range(op.r + row, static_cast<int64_t>(H) * (2 * Storage<DT>::UNITS));
    grid_dependency_wait();
    grid_launch_dependents();

    // the residual is consumed last but requested first, together with the first group of partials
    // (LATE_R: after the last one)
    Pack<UV> pr[VPT];
    auto fetch_residual = [&] {
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const int v = threadIdx.x + i * blockDim.x;
            if (v < nvec) pr[i] = load<UV, Ld::Stream>(op.r + row + v * UV);
        }
    };
    if constexpr (!LATE_R) fetch_residual();

    // The loop over groups is unrolled to the largest supported count and left by a break: every copy
    // then has a constant p0 (the first one initialises the sums without a test) and the compiler may
    // move a group's loads above the additions of the group before it.  Measured against the rolled
    // loop at [8192, 4096], L2-cold: 54.1 -> 50.8 us with 2 partials, 74.5 -> 71.8 us with 4,
    // 113.8 -> 111.8 us with 8.
    float s[VPT][VEC];
#pragma unroll
    for (int p0 = 0; p0 < kMaxParts; p0 += GROUP) {
        if (p0 >= n) break;
        Pack<UV> px[GROUP][VPT];
#pragma unroll
        for (int g = 0; g < GROUP; ++g) {
            if (p0 + g < n) {
                const uint16_t *base = op.part[p0 + g] + row;
#pragma unroll
                for (int i = 0; i < VPT; ++i) {
                    const int v = threadIdx.x + i * blockDim.x;
                    if (v < nvec) px[g][i] = load<UV, Ld::Stream>(base + v * UV);
                }
            }
        }
#pragma unroll
        for (int g = 0; g < GROUP; ++g) {
            if (p0 + g < n) {
#pragma unroll
                for (int i = 0; i < VPT; ++i) {
                    const int v = threadIdx.x + i * blockDim.x;
                    if (v < nvec) {
                        float fx[VEC];
                        widen<DT, VEC>(px[g][i], fx);
                        if (p0 + g == 0) {
#pragma unroll
                            for (int k = 0; k < VEC; ++k) s[i][k] = fx[k];
                        } else {
                            accumulate(s[i], fx);  // rank order: partial p0 + g joins the sum of those before it
                        }
                    }
                }
            }
        }
    }

    if constexpr (LATE_R) fetch_residual();
    float acc = 0.f;
    float2 acc2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < nvec) {
            float fr[VEC];
            widen<DT, VEC>(pr[i], fr);
            add_and_square(s[i], fr, s[i], acc, acc2);  // the residual joins last
            store_to_all<UV>(op.r_out, op.n_r, row + v * UV, narrow<DT, VEC>(s[i]));
        }
    }

    Pack<UV> pw[VPT];
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < nvec) pw[i] = load<UV, Ld::Keep>(weight + v * UV);
    }
    const float total = block_sum(acc + (acc2.x + acc2.y), slots);
    const float rstd = rsqrtf(fmaf(total, inv_H, eps));

#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < nvec) {
            float fw[VEC], fy[VEC];
            widen<DT, VEC>(pw[i], fw);
            scale(s[i], rstd, fw, fy);
            store_to_all<UV>(op.y_out, op.n_y, row + v * UV, narrow<DT, VEC>(fy));
        }
    }
}

// Rows that start at any element (odd widths), all operands at the same place within 32 bytes: body in
// 32-byte vectors, edge one unit per lane of the first two warps, weight shifted, as in
// fused_add_rmsnorm_ragged_kernel; partials and shapes as in the kernel above.  The edge's partials
// are fetched group by group beside the body's.  (The plain loads and stores stay per-thread here too: a
// partial or a destination may be another GPU's memory.)
// Measured L2-cold, bf16, against the 2-, 4- and 8-byte vector kernels: see the launch code.
// With four loads in flight the compiler is asked for no minimum of resident blocks: given one as a minimum it takes 76
// and 134 registers (one and two vectors, 16-bit) instead of 64 and 128 with 16 and 28 bytes of spill, which
// cost a block per SM: 96.8 -> 70.1 us at bf16 [4096, 7167] with 4 partials, 146 -> 113 at [4096, 8191] with 8, 46.6 ->
// 40.6 at [4096, 4099] with 4, 47.7 -> 38.7 at fp32 [2048, 4095] with 4 (12.2 -> 13.6 at bf16 [500, 5123] with 8).
template <int DT, int VPT, int GROUP, bool LATE_R = false>
__global__ void __launch_bounds__(LATE_R ? kAllreduceLateThreads : VPT == 4 ? 512 : allreduce_reg_max_threads(16 * VPT, GROUP),
                                  LATE_R ? 2 : GROUP == 4 ? 0 : 1)
fused_allreduce_add_rmsnorm_ragged_kernel(const __grid_constant__ AllreduceOperands op,
                                          const uint16_t *__restrict__ weight, int H, float eps, float inv_H, LaunchPad<40>) {
    constexpr int UV = 16, UNITS = Storage<DT>::UNITS, VEC = UV / UNITS;
    constexpr bool EDGE_LAST = GROUP == 4 || GROUP == 1 || LATE_R, EARLY_W = GROUP > 4;
    __shared__ __align__(16) float slots[kMaxWarps];
    const int units = H * UNITS;
    const int64_t row = static_cast<int64_t>(blockIdx.x) * units;
    const int n = op.n_parts;
    if (threadIdx.x == 0) prefetch_l2_range(op.r + row, static_cast<int64_t>(units) * 2);
    const RaggedRow g = ragged_row<UNITS>(op.r + row, weight, units, static_cast<int>(threadIdx.x));
    const int64_t body = row + g.first;
    grid_dependency_wait();
    grid_launch_dependents();

    Pack<UV> pr[VPT];
    Pack<UNITS> er, ew;
    auto fetch_residual = [&] {
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const int v = threadIdx.x + i * blockDim.x;
            if (v < g.nvec) pr[i] = load<UV, Ld::Stream>(op.r + body + v * UV);
        }
    };
    if constexpr (!LATE_R) fetch_residual();
    if (!EDGE_LAST && g.edge >= 0) {
        er = load<UNITS, Ld::Stream>(op.r + row + g.edge);
        ew = load<UNITS, Ld::Keep>(weight + g.edge);
    }
    float s[VPT][VEC], es[1] = {0.f};
#pragma unroll
    for (int p0 = 0; p0 < kMaxParts; p0 += GROUP) {
        if (p0 >= n) break;
        Pack<UV> px[GROUP][VPT];
        Pack<UNITS> ex[GROUP];
#pragma unroll
        for (int q = 0; q < GROUP; ++q) {
            if (p0 + q < n) {
                const uint16_t *base = op.part[p0 + q];
#pragma unroll
                for (int i = 0; i < VPT; ++i) {
                    const int v = threadIdx.x + i * blockDim.x;
                    if (v < g.nvec) px[q][i] = load<UV, Ld::Stream>(base + body + v * UV);
                }
                if (!EDGE_LAST && g.edge >= 0) ex[q] = load<UNITS, Ld::Stream>(base + row + g.edge);
            }
        }
#pragma unroll
        for (int q = 0; q < GROUP; ++q) {
            if (p0 + q < n) {
#pragma unroll
                for (int i = 0; i < VPT; ++i) {
                    const int v = threadIdx.x + i * blockDim.x;
                    if (v < g.nvec) {
                        float fx[VEC];
                        widen<DT, VEC>(px[q][i], fx);
                        if (p0 + q == 0) {
#pragma unroll
                            for (int k = 0; k < VEC; ++k) s[i][k] = fx[k];
                        } else {
                            accumulate(s[i], fx);
                        }
                    }
                }
                if (!EDGE_LAST && g.edge >= 0) {
                    float fx[1];
                    widen<DT, 1>(ex[q], fx);
                    if (p0 + q == 0) es[0] = fx[0];
                    else accumulate(es, fx);
                }
            }
        }
    }

    if constexpr (LATE_R) fetch_residual();
    float acc = 0.f;
    float2 acc2 = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int v = threadIdx.x + i * blockDim.x;
        if (v < g.nvec) {
            float fr[VEC];
            widen<DT, VEC>(pr[i], fr);
            add_and_square(s[i], fr, s[i], acc, acc2);
            store_to_all<UV>(op.r_out, op.n_r, body + v * UV, narrow<DT, VEC>(s[i]));
        }
    }
    if (EDGE_LAST && g.edge >= 0) {
        er = load<UNITS, Ld::Stream>(op.r + row + g.edge);
        ew = load<UNITS, Ld::Keep>(weight + g.edge);
#pragma unroll
        for (int p0 = 0; p0 < kMaxParts; p0 += 8) {
            if (p0 >= n) break;
            Pack<UNITS> ex[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (p0 + q < n) ex[q] = load<UNITS, Ld::Stream>(op.part[p0 + q] + row + g.edge);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (p0 + q < n) {
                    float fx[1];
                    widen<DT, 1>(ex[q], fx);
                    if (p0 + q == 0) es[0] = fx[0];
                    else accumulate(es, fx);
                }
            }
        }
    }
    if (g.edge >= 0) {
        float fr[1];
        widen<DT, 1>(er, fr);
        add_and_square(es, fr, es, acc, acc2);
        store_to_all<UNITS>(op.r_out, op.n_r, row + g.edge, narrow<DT, 1>(es));
    }
    auto store_y = [&](int at, const auto &v) {
        store_to_all<std::decay_t<decltype(v)>::UNITS_PER_PACK>(op.y_out, op.n_y, row + at, v);
    };
    ASTRA_FOR_SHIFT(g.shift, UNITS,
                    (ragged_finish<SHIFT, DT, VPT, EARLY_W>(g, weight, acc + (acc2.x + acc2.y), eps, inv_H, slots, s, es, ew,
                                                          store_y)))
}

// Launch shapes of the two kernels in their 32-byte forms.  Measured L2-cold against the 16-byte form at [8192, 4096]: 50.6 -> 49.2 us with 2 partials, 70.8 -> 66.6 us with 4,
// 110.9 -> 104.7 us with 8; at [1024, 4096]: 8.3 -> 7.7, 10.9 -> 10.3, 16.2 -> 15.9 us.
//
// Five shapes: one or two vectors per thread (16 or 32 units), two or four partial loads in flight
// (four only from four partials on), and two of each with the residual requested last.  What decides
// between them is how many bytes of loads an SM has in flight, i.e. resident blocks x threads x bytes per
// thread, with the blocks that are resident (resident_blocks, registers as compiled for sm_100a).  The measurements across H = 2048 ... 16384 fit one rule: take the first shape, in the
// order below, that keeps about 90 KB in flight per SM; if none does, the one with the most.  Examples:
// H = 4096 takes one vector and four in flight (three 256-thread blocks per SM); H = 8192 with four
// in flight would leave one 512-thread block per SM, so it takes two vectors in 256-thread blocks
// (78.8 -> 68.0 us with 4 partials, 117.3 -> 105.6 us with 8); H = 10240 with two in flight takes two
// vectors in 320-thread blocks (two per SM) rather than one 640-thread block (61.6 against 76.7 us);
// H = 11008 ... 14336 take the late residual (79.7 -> 67.9 us at [4096, 11008] with 2 partials, more at the
// kernel; but 2.7 against 3.2 us at [16, 11008], where every SM has one row at most); H = 16384 takes one vector in
// one 1024-thread block (143.1 against 155.8 us with 4 partials).
// Binary32 rows need fewer registers (5120 elements take one vector in two 640-thread blocks: 25.1 -> 23.1 us at
// [1024, 5120] with 4 partials).
// Binary32 rows of more than 16384 units take four vectors per thread, one load in flight, in one block
// of up to 512 threads per SM, instead of two sweeps: 73.5 -> 52.6, 105.8 -> 73.5, 191 -> 112.5 us at [1024, 16384]
// with 2 / 4 / 8 partials (48.6 / 68.1 / 107 us at 6.9 TB/s), 17.5 -> 9.5 us at [16, 16384] with 8.
struct WideShape {
    int vpt, group, regs, max_threads, min_threads;
    bool late = false;  // the residual is requested after the partials
};
constexpr int kStreamGroup = 2;  // partial loads in flight: long streams,
constexpr int kDeepGroup = 8;    // and few rows
#ifndef ASTRA_ALLREDUCE_DEEP_QUEUE_ROWS
#define ASTRA_ALLREDUCE_DEEP_QUEUE_ROWS 128
#endif
constexpr int64_t kDeepQueueRows = ASTRA_ALLREDUCE_DEEP_QUEUE_ROWS;
constexpr int64_t kOneBlockRows = 148;  // rows up to which every SM of a B200 has one block at most
constexpr int kWideShapeCount = 5;
constexpr WideShape kWideShapes[2][kWideShapeCount] = {
    {{1, 4, 72, 512, 128}, {2, 4, 128, 256, 64}, {1, 2, 56, 1024, 128}, {2, 2, 96, 512, 64}, {2, 2, 72, kAllreduceLateThreads, 64, true}},
    {{1, 4, 64, 512, 128}, {2, 4, 112, 256, 64}, {1, 2, 48, 1024, 128}, {2, 2, 80, 512, 64}, {2, 2, 64, kAllreduceLateThreads, 64, true}}};  // binary32
// The same shapes of the ragged kernel, with its registers.
constexpr WideShape kRaggedShapes[2][kWideShapeCount] = {
    {{1, 4, 64, 512, 64}, {2, 4, 128, 256, 64}, {1, 2, 64, 1024, 64}, {2, 2, 112, 512, 64}, {2, 2, 72, kAllreduceLateThreads, 64, true}},
    {{1, 4, 64, 512, 64}, {2, 4, 120, 256, 64}, {1, 2, 56, 1024, 64}, {2, 2, 96, 512, 64}, {2, 2, 64, kAllreduceLateThreads, 64, true}}};
constexpr int64_t kWideBytesInFlight = 90 * 1024;

// Shape for T rows of `units` 16-bit units with n_parts partials; vpt = 0 where none applies (rows too narrow for
// 128-thread blocks, ragged ones for 64, or too wide).
struct AllreduceShape {
    int vpt = 0, group = 0, threads = 0;
    bool late = false;
};
inline AllreduceShape allreduce_wide_shape(int64_t T, int units, int n_parts, bool binary32, bool ragged) {
    const int nvec = units / 16;  // whole vectors (a ragged row has no more inside it)
    auto threads_for = [&](int vpt) { return ((nvec + vpt - 1) / vpt + 31) / 32 * 32; };
    // Few rows and more than four partials: all of a row's partials in one round trip (eight loads in
    // flight, one vector per thread); with so few blocks the registers that costs do not matter.
    // Device time from a graph, 8 partials, against the streaming shapes: 3.19 -> 2.70 us at [16, 4096],
    // 4.17 -> 3.41 us at [16, 8192], 4.12 -> 3.85 us at [128, 4096]; slower from 192 rows on (7.93 -> 8.89 us
    // at [192, 8192]).  With up to four partials the streaming shapes are the fastest at every row
    // count (1.65 / 1.98 us at [16, 4096] with 2 / 4 partials, where the 16-byte shapes took 2.08 / 2.40).
    // (The ragged kernel's four-in-flight shape fetches its edge last, so there four partials count as many.)
    if (T <= kDeepQueueRows && n_parts > (ragged ? 3 : 4) && threads_for(1) >= (ragged ? 64 : 128) &&
        threads_for(1) <= allreduce_reg_max_threads(16, kDeepGroup))
        return {1, kDeepGroup, threads_for(1)};
    // Blocks without a row are not resident: binary32 rows of 11008 units keep one vector per thread up to 148 rows
    // (4.7 against 6.5 us at [16, 6144] with 8 partials), and threads beyond the row's vectors have no loads.  The
    // ragged kernel's edge wants both all the same (3.3 against 4.9 us at bf16 [500, 1059] with 2, 2.9 against 4.1
    // us at [150, 1603]), but no late residual for blocks that are not there (3.4 against 3.9 us at fp32 [150, 3202]).
    const int64_t rows_per_sm = (T + kOneBlockRows - 1) / kOneBlockRows;
    AllreduceShape best;
    int64_t best_bytes = 0;
    for (const WideShape &sh : (ragged ? kRaggedShapes : kWideShapes)[binary32]) {
        if (sh.group > kStreamGroup && n_parts < sh.group) continue;
        if (sh.late && T <= kOneBlockRows) continue;  // a second block per SM has no row to work on then
        const int threads = threads_for(sh.vpt);
        if (threads > sh.max_threads || threads < sh.min_threads) continue;
        int64_t resident = resident_blocks(sh.regs, threads);
        if ((!ragged || sh.late) && resident > rows_per_sm) resident = rows_per_sm;
        const int64_t vectors = ragged ? threads * sh.vpt : nvec;
        const int64_t bytes = resident * vectors * (sh.group + (sh.late ? 0 : 1)) * 32;
        if (bytes > best_bytes) {
            best = {sh.vpt, sh.group, threads, sh.late};
            best_bytes = bytes;
        }
        if (bytes >= kWideBytesInFlight) break;  // the first shape that reaches it is also the largest so far
    }
    if (best.vpt == 0 && binary32 && nvec > 1024 && threads_for(4) <= allreduce_reg_max_threads(64, 1))
        return {4, 1, threads_for(4)};
    return best;
}

// Do T rows of `units` units that start at no 16-byte boundary stay with the 2-, 4- or 8-byte forms (vec = 1, 2, 4
// units), or do they go to the ragged kernel?  Only 8-byte forms are ever the faster, and short rows of 4-byte ones
// that are few.  Their smaller code starts sooner and they keep eight loads in flight up to 296 rows, which counts
// while a row is short or the SMs have few.  Narrow against ragged, bf16: 2.6 and 4.1 us at [150, 1060] with 8
// partials, 3.0 and 4.0 us at [150, 3076] with 4, 3.4 and 4.1 us at [800, 1060] with 2, 18.4 and 21.3 us at [3000, 3588]
// with 2; but 4.4 and 3.8 us at [150, 4100] with 4, 6.3 and 4.9 us at [300, 2084] with 8, 25.7 and 22.9 us at [1500, 5124] with 4, and
// anything from there on.  binary32: 2.2 and 2.6 us at [150, 802] with 2, 3.1 and 3.7 us at [150, 602] with 8; 4.4
// and 2.9 us at [150, 2050] with 4, 9.9 and 8.6 us at [1500, 2050] with 2; from 10241 to 16384 units the narrow forms are
// the faster throughout (41.2 against 45.9 us at [1024, 8190] with 4).
inline bool allreduce_keeps_narrow(int64_t T, int units, int n_parts, bool binary32, int vec) {
    const bool few = T <= kOneBlockRows, several = T <= 2 * kOneBlockRows, short_rows = units < 4096;
    if (vec != 4) return vec == 2 && !binary32 && units < 1536 && n_parts < 4 && T <= 160;
    if (!binary32) {
        if (n_parts < 4) return T <= 512 || short_rows;
        if (few) return units <= 8192;
        if (n_parts < 6) return (short_rows && T <= 512) || units < 2560;
        return short_rows && several;
    }
    if (units > 10240) return units <= 16384;
    if (few) return n_parts < 4 || short_rows || units > 8704 || (T > 128 && (n_parts < 6 || units < 8192));
    if (n_parts == 2) return (units < 8192 && T <= (units < 4608 ? 400 : 200)) || (short_rows && T <= 512) || units < 2048;
    if (n_parts < 4) return (short_rows && T <= 512) || units < 2048;
    return (short_rows && several) || (n_parts < 6 && units < 2560);
}

// The rank-order sum of one vector position, GROUP partial loads in flight at a time.
template <int DT, int VEC, int GROUP>
__device__ __forceinline__ void rank_order_sum(const AllreduceOperands &op, int64_t at, float (&s)[VEC]) {
    constexpr int UV = VEC * Storage<DT>::UNITS;
    const int n = op.n_parts;
    const Pack<UV> pr = load<UV, Ld::Stream>(op.r + at);
#pragma unroll
    for (int p0 = 0; p0 < kMaxParts; p0 += GROUP) {  // unrolled and left by a break, as in the kernel above
        if (p0 >= n) break;
        Pack<UV> px[GROUP];
#pragma unroll
        for (int g = 0; g < GROUP; ++g)
            if (p0 + g < n) px[g] = load<UV, Ld::Stream>(op.part[p0 + g] + at);
#pragma unroll
        for (int g = 0; g < GROUP; ++g) {
            if (p0 + g < n) {
                float fx[VEC];
                widen<DT, VEC>(px[g], fx);
                if (p0 + g == 0) {
#pragma unroll
                    for (int k = 0; k < VEC; ++k) s[k] = fx[k];
                } else {
                    accumulate(s, fx);
                }
            }
        }
    }
    float fr[VEC];
    widen<DT, VEC>(pr, fr);
    accumulate(s, fr);
}

// Any width and any vector size: two sweeps over the row.  The first forms the sums and their
// squares and writes nothing; the second forms the same sums again (the partials now come from L2
// where they fit) and writes both outputs, so the in-place residual cannot disturb the reduction.
template <int DT, int VEC, int GROUP>
__global__ void __launch_bounds__(1024)
fused_allreduce_add_rmsnorm_twopass_kernel(const __grid_constant__ AllreduceOperands op,
                                           const uint16_t *__restrict__ weight, int H, float eps, float inv_H, LaunchPad<40>) {
    constexpr int UV = VEC * Storage<DT>::UNITS;
    __shared__ __align__(16) float slots[kMaxWarps];
    const int nvec = H / VEC;
    const int64_t row = static_cast<int64_t>(blockIdx.x) * H * Storage<DT>::UNITS;
    grid_dependency_wait();
    grid_launch_dependents();

    float acc = 0.f;
    for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
        float s[VEC];
        rank_order_sum<DT, VEC, GROUP>(op, row + static_cast<int64_t>(v) * UV, s);
#pragma unroll
        for (int k = 0; k < VEC; ++k) acc = fmaf(s[k], s[k], acc);
    }
    const float total = block_sum(acc, slots);
    const float rstd = rsqrtf(fmaf(total, inv_H, eps));

    for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
        const int64_t at = row + static_cast<int64_t>(v) * UV;
        float s[VEC], fw[VEC], fy[VEC];
        rank_order_sum<DT, VEC, GROUP>(op, at, s);
        widen<DT, VEC>(load<UV, Ld::Keep>(weight + static_cast<int64_t>(v) * UV), fw);
#pragma unroll
        for (int k = 0; k < VEC; ++k) fy[k] = s[k] * rstd * fw[k];
        store_to_all<UV>(op.r_out, op.n_r, at, narrow<DT, VEC>(s));
        store_to_all<UV>(op.y_out, op.n_y, at, narrow<DT, VEC>(fy));
    }
}

}  // namespace astra
