// Runs of calls: several calls of one kind and shape in one launch, for sequences that are captured into a
// graph.  A decode-sized call is a chain of latencies (launch, first bytes, reduction, completion: 1.4 us at
// [16, 4096] for 0.1 us of work), and calls that follow one another on a shared tensor pay it one after the
// other.  All three operations work on rows (the norm) or vectors (the others) that depend on nothing else, so
// the threads that own one take it through all calls of the run: what a later call reads of an earlier one (the
// residual) or overwrites (a shared output) then stays within a thread, in order, and the next calls' operands
// are on their way while this one's are worked on.
//
// The launch code admits a call to a run only where nothing else is shared: what any call of the run reads is
// written by none of the others (the residual apart), and two written tensors are the same or disjoint.
#pragma once

#include "fused_add_rmsnorm.cuh"
#include "merge_attn_states_lse.cuh"
#include "silu_and_mul.cuh"

namespace astra {

constexpr int kMaxRun = 64;  // calls of one launch: their addresses are kernel parameters

// Polls of one wait of a cluster exchange before it is given up, and the limit that the waits of the exchanges use (a
// test lowers the latter to see what is left of a run whose waits end too early).
constexpr int kWaitPolls = 1 << 16;
#ifndef ASTRA_RUN_WAIT_POLLS
#define ASTRA_RUN_WAIT_POLLS kWaitPolls
#endif

// ---- fused_add_rmsnorm: calls on one residual ----------------------------------------------------------------
struct RmsnormRun {
    uint16_t *x[kMaxRun];
    const uint16_t *w[kMaxRun];
    uint16_t *r;
    int n, H, blocks;
    float eps, inv_H;
};

// The blocks of a run: `blocks` of them share a row (a cluster where there are several), each thread has one vector of
// `uvec` units.  threads = 0: no form for this size.
// Spreading a row pays while SMs would be idle: one SM moves a row's 24 KB per call (x, weight, y at H = 4096) at 52
// GB/s.  64 calls in one launch, from a graph, us, with 1 / 2 / 4 / 8 blocks per row: 43 / 24.6 / 22.6 / 26.6 at
// [16, 4096], 45 / 24.8 / 28.7 / 32.8 at [64, 4096], 59 / 47 / 28.7 / 34 at [16, 8192]; one
// by one 86, 115 and 113.
// Rows of up to 8192 units (16-bit elements; half as many of binary32); wider ones, and widths that are not whole
// vectors, have no form and are launched one by one.  Rows of fewer vectors than a cluster has threads leave some of its
// blocks without any.
constexpr int64_t kSms = 148;
struct NormRunShape {
    int blocks = 0, threads = 0, uvec = 0;
};
inline NormRunShape norm_run_shape(int64_t T, int64_t units, int vec) {
    auto threads_for = [&](int uvec, int blocks) {
        return (units / uvec + blocks * 32 - 1) / (blocks * 32) * 32;
    };
    auto shape = [&](int uvec, int blocks) { return NormRunShape{blocks, static_cast<int>(threads_for(uvec, blocks)), uvec}; };
    if (vec < 8 || units % vec != 0) return {};
    if (T <= kSms / 4 && threads_for(8, 4) <= 256) return shape(8, 4);
    if (T <= kSms / 2 && threads_for(8, 2) <= 256) return shape(8, 2);
    if (threads_for(8, 1) <= 512) return shape(8, 1);
    if (vec == 16 && threads_for(16, 1) <= 512) return shape(16, 1);
    return {};
}

// Sums of K values over the warp (K a power of two up to 32); lane l receives that of value l * K / 32.  Each of the
// first log2 K exchanges halves the number of values that a lane still carries.
template <int K> __device__ __forceinline__ float warp_sums(float (&v)[K]) {
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int have = K; have > 1; have >>= 1, off >>= 1) {
        const bool high = lane & off;
#pragma unroll
        for (int k = 0; k < have / 2; ++k) {
            const float keep = high ? v[k + have / 2] : v[k], give = high ? v[k] : v[k + have / 2];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, off);
        }
    }
#pragma unroll
    for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    return v[0];
}

// Exchange of sums within a cluster: a store into a block's shared memory that counts its bytes on that block's
// barrier.  (A cluster barrier instead would have to wait for the block's global stores as well.)
__device__ __forceinline__ uint32_t shared_address(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ uint32_t in_block(uint32_t address, int rank) {
    uint32_t at;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(address), "r"(rank));
    return at;
}
__device__ __forceinline__ void store_counted(uint32_t address, float v, uint32_t barrier) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(address), "f"(v), "r"(barrier) : "memory");
}
__device__ __forceinline__ void init_barrier(uint32_t barrier) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(barrier) : "memory");
}
__device__ __forceinline__ void expect_bytes(uint32_t barrier, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(barrier), "r"(bytes) : "memory");
}
// Waits for the barrier's phase; false if it has not ended after so many polls.
__device__ __forceinline__ bool wait_counted(uint32_t barrier, uint32_t phase, int polls) {
    for (int i = 0; i < polls; ++i) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
            : "=r"(done) : "r"(barrier), "r"(phase) : "memory");
        if (done) return true;
    }
    return false;
}

// The row's residual stays in registers from the first call to the last.  The calls are taken K at a time: their loads
// are in flight together, and their sums of squares, which nothing later in the chain of residuals waits for,
// go through the block or cluster in one exchange: every warp stores its K sums where all can read them
// (in a cluster, into every block's shared memory), and after one wait every warp adds up all warps' sums in the same
// order.  The next exchange uses the other half of `slots`; nobody can be two exchanges ahead of another.
//
// In a cluster the wait is bounded.  A warp whose wait runs out has its share of the present and of all later normalised
// rows set to NaN, stores nothing more into other blocks and arms no barrier again (one whose phase has not ended
// must not be); the other warps of the row, which then lack its sums, run out at the next exchange and do the same.
// Nobody reads sums of two exchanges that way, and the residual, which needs no sums, is as it should be.  Before it
// leaves, such a warp waits once more, up to the full limit, for the stores that it gave up on.
// 1.34 -> 0.35 us per call at [16, 4096].  Also tried: one call at a time with the next x and weight loaded ahead (0.74
// to 0.9 us with 128 to 512 threads: the loads share the few scoreboards, so a wait for one waits for the latest), and
// a cluster barrier for the exchange (0.41 us: its release waits for the block's stores to global memory).
template <int DT, int VEC, int K, int THREADS, bool CLUSTER>
__global__ void __launch_bounds__(THREADS) fused_add_rmsnorm_run_kernel(const __grid_constant__ RmsnormRun run) {
    constexpr int UV = VEC * Storage<DT>::UNITS, SHARE = 32 / K;  // lanes that carry one of the K sums
    __shared__ float slots[2][K][kMaxWarps];
    __shared__ __align__(8) uint64_t barriers[2];
    const int blocks = CLUSTER ? run.blocks : 1, rank = blockIdx.x % blocks;
    const int n = run.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int64_t units = static_cast<int64_t>(run.H) * Storage<DT>::UNITS, row = blockIdx.x / blocks * units;
    const int v = rank * blockDim.x + threadIdx.x, at = v * UV;
    const bool mine = v < run.H / VEC;
    if (v == 0) prefetch_l2_range(run.r + row, units * 2);
    if (v < n) prefetch_l2_range(run.x[v] + row, units * 2);
    if constexpr (CLUSTER) {
        if (threadIdx.x == 0) {
            init_barrier(shared_address(&barriers[0]));
            init_barrier(shared_address(&barriers[1]));
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    }
    grid_dependency_wait();

    Pack<UV> pr, px[K], pw[K];
    auto fetch_x = [&](int i0) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (i0 + k < n) px[k] = load<UV, Ld::Stream>(run.x[i0 + k] + row + at);
    };
    if (mine) {
        pr = load<UV, Ld::Stream>(run.r + row + at);
        fetch_x(0);
    }
    if constexpr (CLUSTER) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");  // every block's barriers are ready
    int gave_up = -1;  // the exchange whose wait ran out
    float s[K][VEC];
    for (int i0 = 0, exchange = 0; i0 < n; i0 += K, ++exchange) {
        const int half = exchange & 1;
        float acc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            float one = 0.f;
            float2 acc2 = make_float2(0.f, 0.f);
            if (mine && i0 + k < n) {
                float fx[VEC], fr[VEC];
                widen<DT, VEC>(px[k], fx);
                widen<DT, VEC>(pr, fr);
                add_and_square(fx, fr, s[k], one, acc2);
                pr = narrow<DT, VEC>(s[k]);
            }
            acc[k] = one + (acc2.x + acc2.y);
        }
        if (mine) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (i0 + k < n) pw[k] = load<UV, Ld::Keep>(run.w[i0 + k] + at);
            fetch_x(i0 + K);
        }
        const float partial = warp_sums<K>(acc);
        float *slot = &slots[half][lane / SHARE][rank * nwarps + warp];
        if constexpr (CLUSTER) {
            if (gave_up < 0) {
                const uint32_t barrier = shared_address(&barriers[half]);
                if (threadIdx.x == 0) expect_bytes(barrier, blocks * nwarps * K * static_cast<uint32_t>(sizeof(float)));
                for (int p = lane % SHARE; p < blocks; p += SHARE)
                    store_counted(in_block(shared_address(slot), p), partial, in_block(barrier, p));
                if (!__all_sync(0xffffffffu, wait_counted(barrier, (exchange >> 1) & 1, ASTRA_RUN_WAIT_POLLS))) gave_up = exchange;
            }
        } else {
            if (lane % SHARE == 0) *slot = partial;
            __syncthreads();
        }
        float total = 0.f;  // of call i0 + lane / SHARE
        for (int w = lane % SHARE; w < blocks * nwarps; w += SHARE) total += slots[half][lane / SHARE][w];
#pragma unroll
        for (int off = SHARE / 2; off > 0; off >>= 1) total += __shfl_xor_sync(0xffffffffu, total, off);
        const float rstd = gave_up < 0 ? rsqrtf(fmaf(total, run.inv_H, run.eps)) : __int_as_float(0x7fc00000);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float rk = __shfl_sync(0xffffffffu, rstd, k * SHARE);
            if (mine && i0 + k < n) {
                float fw[VEC], fy[VEC];
                widen<DT, VEC>(pw[k], fw);
                scale(s[k], rk, fw, fy);
                store<UV, St::Stream>(run.x[i0 + k] + row + at, narrow<DT, VEC>(fy));
            }
        }
    }
    grid_launch_dependents();
    if (mine) store<UV, St::Stream>(run.r + row + at, pr);
    if constexpr (CLUSTER) {  // no block leaves while another may still store into its shared memory
        if (gave_up >= 0) wait_counted(shared_address(&barriers[gave_up & 1]), (gave_up >> 1) & 1, kWaitPolls);
        asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
        asm volatile("barrier.cluster.wait;" ::: "memory");
    }
}

// ---- silu_and_mul ----------------------------------------------------------------------------------------------
// Elementwise: a thread takes its 16-byte vector through all calls, kRunGroup of them loaded at a time and the next
// group asked for before the present one is worked on.  1.1 -> 0.32 us per call at [16, 14336], 32 calls.
constexpr int kRunGroup = 4, kRunThreads = 128;

struct SiluRun {
    const uint16_t *in[kMaxRun];
    uint16_t *out[kMaxRun];
    int64_t D;  // in units
    int n;
    uint32_t total_vecs;
    FastDiv nvec;
};

// load(i, k, half) fetches call i as the k-th of a half's group; finish(i, k, half) works on it and stores.
template <typename LOAD, typename FINISH> __device__ __forceinline__ void run_in_groups(int n, LOAD load, FINISH finish) {
#pragma unroll
    for (int k = 0; k < kRunGroup; ++k)
        if (k < n) load(k, k, 0);
    for (int i0 = 0; i0 < n; i0 += 2 * kRunGroup) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int first = i0 + half * kRunGroup;
#pragma unroll
            for (int k = 0; k < kRunGroup; ++k)
                if (first + kRunGroup + k < n) load(first + kRunGroup + k, k, half ^ 1);
#pragma unroll
            for (int k = 0; k < kRunGroup; ++k)
                if (first + k < n) finish(first + k, k, half);
        }
    }
}

template <int DT> __global__ void __launch_bounds__(kRunThreads) silu_and_mul_run_kernel(const __grid_constant__ SiluRun run) {
    constexpr int UV = 8;
    const uint32_t v = blockIdx.x * kRunThreads + threadIdx.x;
    const uint32_t row = run.nvec.div(v), col = v - row * run.nvec.d;
    const int64_t gate = row * (2 * run.D) + col * UV, out = static_cast<int64_t>(v) * UV;
    grid_dependency_wait();
    if (v < run.total_vecs) {
        Pack<UV> a[2][kRunGroup], b[2][kRunGroup];
        run_in_groups(
            run.n,
            [&](int i, int k, int half) {
                a[half][k] = load<UV, Ld::StreamReadOnly>(run.in[i] + gate);
                b[half][k] = load<UV, Ld::StreamReadOnly>(run.in[i] + gate + run.D);
            },
            [&](int i, int k, int half) {
                store<UV, St::Stream>(run.out[i] + out, silu_mul_pack<DT, UV>(a[half][k], b[half][k]));
            });
    }
    grid_launch_dependents();
}

// ---- merge_attn_states_lse: likewise; 1.15 -> 0.39 us per call at [16, 32, 128], 32 calls --------------------------
struct MergeRun {
    const uint16_t *v_a[kMaxRun], *v_b[kMaxRun];
    const float *lse_a[kMaxRun], *lse_b[kMaxRun];
    uint16_t *v_out[kMaxRun];
    float *lse_out[kMaxRun];  // or null
    int n;
    uint32_t total_vecs;
    FastDiv nvec;
};

template <int DT>
__global__ void __launch_bounds__(kRunThreads) merge_attn_states_lse_run_kernel(const __grid_constant__ MergeRun run) {
    constexpr int UV = 8;
    const uint32_t v = blockIdx.x * kRunThreads + threadIdx.x;
    const uint32_t row = run.nvec.div(v);
    const bool first_of_row = v == row * run.nvec.d;
    const int64_t at = static_cast<int64_t>(v) * UV;
    grid_dependency_wait();
    if (v < run.total_vecs) {
        Pack<UV> a[2][kRunGroup], b[2][kRunGroup];
        float sa[2][kRunGroup], sb[2][kRunGroup];
        run_in_groups(
            run.n,
            [&](int i, int k, int half) {
                a[half][k] = load<UV, Ld::Stream>(run.v_a[i] + at);
                b[half][k] = load<UV, Ld::Stream>(run.v_b[i] + at);
                sa[half][k] = run.lse_a[i][row];
                sb[half][k] = run.lse_b[i][row];
            },
            [&](int i, int k, int half) {
                const MergeWeights mw = merge_weights(sa[half][k], sb[half][k]);
                store<UV, St::Stream>(run.v_out[i] + at, merge_packs<DT, UV>(mw, a[half][k], b[half][k]));
                if (first_of_row && run.lse_out[i] != nullptr) run.lse_out[i][row] = mw.lse;
            });
    }
    grid_launch_dependents();
}

}  // namespace astra
