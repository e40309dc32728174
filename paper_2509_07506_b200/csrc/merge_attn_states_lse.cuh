// merge_attn_states_lse (Astra paper, Table 1, Kernel 1):
//     V_out = (e^{Sa} Va + e^{Sb} Vb) / (e^{Sa} + e^{Sb}),   S_out = log(e^{Sa} + e^{Sb}).
//
// HBM-bound: per (token, head) row of D elements, 2*D*2 bytes are read and D*2 written, plus three
// 4-byte scores.  The two mixing weights depend only on the row, so each thread derives them once
// for the vector(s) it owns (the paper's hoisting of the exponentials out of the element loop); the
// element work is one multiply and one fused multiply-add.
#pragma once

#include "vec.cuh"

namespace astra {

struct MergeWeights {
    float wa, wb;   // normalised weights of the two states
    float lse;      // merged score
    bool use_a, use_b;
};

// m = max(Sa, Sb); with t = e^{min - max} in [0, 1]: weight of the larger = 1/(1+t), of the
// smaller = t/(1+t), S_out = m + log(1+t).  A score of -inf gives t = 0 exactly, so the other state
// passes through with weight exactly 1; its own V is not used at all.  Both -inf: empty result.
__device__ __forceinline__ MergeWeights merge_weights(float sa, float sb) {
    MergeWeights r;
    const float m = fmaxf(sa, sb);
    const float lo = fminf(sa, sb);
    if (m == -INFINITY) {  // both states empty
        r.wa = 0.f; r.wb = 0.f; r.lse = -INFINITY; r.use_a = false; r.use_b = false;
        return r;
    }
    // t in [0, 1]; exactly 0 for lo = -inf, exactly 1 for lo = m.  Non-flushing ex2, so a weight
    // below 2^-126 is still a (subnormal) weight rather than zero.
    float t;
    asm("ex2.approx.f32 %0, %1;" : "=f"(t) : "f"((lo - m) * 1.4426950408889634f));
    const float inv = __fdividef(1.0f, 1.0f + t);
    const float w_hi = inv, w_lo = t * inv;
    const bool a_is_hi = sa >= sb;
    r.wa = a_is_hi ? w_hi : w_lo;
    r.wb = a_is_hi ? w_lo : w_hi;
    // log(1 + t) with 1 + t in [1, 2]: lg2.approx is within about 2^-22 absolute there
    float l2;
    asm("lg2.approx.f32 %0, %1;" : "=f"(l2) : "f"(1.0f + t));
    r.lse = fmaf(l2, 0.6931471805599453f, m);
    // +inf or NaN scores are outside the domain (e^{S} / e^{S} = inf / inf): everything becomes NaN.
    if (!(m < INFINITY) || sa != sa || sb != sb) { r.wa = r.wb = r.lse = __int_as_float(0x7fc00000); }
    r.use_a = !(r.wa == 0.f);
    r.use_b = !(r.wb == 0.f);
    return r;
}

// The blend of two vectors of UV units.  A zero-weight side is dropped, not multiplied: its payload may be
// Inf/NaN garbage.
template <int DT, int UV>
__device__ __forceinline__ Pack<UV> merge_packs(const MergeWeights &mw, const Pack<UV> &a, const Pack<UV> &b) {
    constexpr int VEC = UV / Storage<DT>::UNITS;
    float fa[VEC], fb[VEC], fo[VEC];
    widen<DT, VEC>(a, fa);
    widen<DT, VEC>(b, fb);
#pragma unroll
    for (int i = 0; i < VEC; ++i) {
        const float ta = mw.use_a ? fa[i] * mw.wa : 0.f;
        fo[i] = mw.use_b ? fmaf(fb[i], mw.wb, ta) : ta;
    }
    return narrow<DT, VEC>(fo);
}

// Strides of one [T, Hh, D] value tensor (in 16-bit units) or one [T, Hh] score tensor (in floats);
// D is contiguous.
struct MergeStrides {
    int64_t va_t, va_h, vb_t, vb_h, vo_t, vo_h;  // values: token and head strides
    int64_t sa_t, sa_h, sb_t, sb_h, so_t, so_h;  // scores: token and head strides
};

// Flat indexing over vectors of VEC elements: vector v belongs to row = v / nvec (row = token*Hh+head).
template <int DT, int VEC, int UNROLL, int THREADS, Ld LDH = Ld::Stream, St STH = St::Stream, bool PREFETCH = true>
__global__ void __launch_bounds__(THREADS)
merge_attn_states_lse_kernel(uint16_t *v_out, float *lse_out,
                             const uint16_t *v_a, const float *lse_a,
                             const uint16_t *v_b, const float *lse_b,
                             uint32_t total_vecs, FastDiv nvec, LaunchPad<24>) {
    constexpr int UV = VEC * Storage<DT>::UNITS;  // 16-bit units per vector
    const uint32_t base = blockIdx.x * (THREADS * UNROLL) + threadIdx.x;
    // Ahead of the dependency wait the block asks for its (contiguous) share of both value tensors to
    // be brought into L2.
    if (PREFETCH && threadIdx.x == 0 && base < total_vecs) {
        const uint32_t n = min(static_cast<uint32_t>(THREADS * UNROLL), total_vecs - base);
        prefetch_l2_range(v_a + static_cast<int64_t>(base) * UV, static_cast<int64_t>(n) * UV * 2);
        prefetch_l2_range(v_b + static_cast<int64_t>(base) * UV, static_cast<int64_t>(n) * UV * 2);
    }
    grid_dependency_wait();
    grid_launch_dependents();
    Pack<UV> a[UNROLL], b[UNROLL];
    float sa[UNROLL], sb[UNROLL];
    uint32_t row[UNROLL];
#pragma unroll
    for (int j = 0; j < UNROLL; ++j) {
        const uint32_t v = base + j * THREADS;
        if (v < total_vecs) {
            row[j] = nvec.div(v);
            // v_out may be exactly v_a or v_b, so these are ordinary (coherent) loads; the thread
            // that reads a vector is the only one that writes it
            a[j] = load<UV, LDH>(v_a + static_cast<int64_t>(v) * UV);
            b[j] = load<UV, LDH>(v_b + static_cast<int64_t>(v) * UV);
            sa[j] = lse_a[row[j]];
            sb[j] = lse_b[row[j]];
        }
    }
#pragma unroll
    for (int j = 0; j < UNROLL; ++j) {
        const uint32_t v = base + j * THREADS;
        if (v < total_vecs) {
            const MergeWeights mw = merge_weights(sa[j], sb[j]);
            store<UV, STH>(v_out + static_cast<int64_t>(v) * UV, merge_packs<DT, UV>(mw, a[j], b[j]));
            if (lse_out != nullptr && v == row[j] * nvec.d) lse_out[row[j]] = mw.lse;
        }
    }
}

}  // namespace astra

namespace astra {

// How the kernel below reads: FEW asks for nothing ahead of the dependency wait; DENSE takes the three value tensors
// as dense [T, Hh, D] (the usual case of head-major scores), addresses their vectors flat, and a block asks for its
// share of each input, one contiguous range, ahead of the wait, as above; ROWS has a thread per row ask for that row.
// A request costs its block time, most where 32 or 64 threads make one each, and pays once the grid's loads queue
// for memory.  FEW against ROWS, L2-cold: 1.17 and 1.97 us at fp32 [8, 32, 64], 1.33 and 2.0 at bf16 [64, 32, 64], 2.0 and 2.35
// at bf16 [64, 32, 128]; but 3.0 and 2.46 at bf16 [1024, 32, 128], 2.87 and 2.55 at fp32 [256, 20, 128].  FEW against DENSE:
// 1.33 and 1.44 at bf16 [16, 40, 128], 1.12 and 1.22 at fp32 [8, 20, 128]; but 2.0 and 1.88 at bf16 [64, 32, 128].
enum class MergeReads { Few, Dense, Rows };
inline MergeReads merge_strided_reads(int64_t blocks, int64_t rows_per_block, bool dense) {
    if (blocks < (dense || rows_per_block <= 8 ? 56 : rows_per_block <= 16 ? 64 : 240)) return MergeReads::Few;
    return dense ? MergeReads::Dense : MergeReads::Rows;
}

// Same computation for arbitrarily strided tensors (head_dim contiguous): row = token * Hh + head is
// split again into (token, head) to address each tensor by its own strides.  This is the form for
// head-major scores ([Hh, T]) or values that are slices of a wider buffer.
template <int DT, int VEC, int UNROLL, int THREADS, MergeReads READS>
__global__ void __launch_bounds__(THREADS)
merge_attn_states_lse_strided_kernel(uint16_t *v_out, float *lse_out,
                                     const uint16_t *v_a, const float *lse_a,
                                     const uint16_t *v_b, const float *lse_b,
                                     uint32_t total_vecs, uint32_t row0, FastDiv nvec, FastDiv heads,
                                     MergeStrides st, LaunchPad<40>) {
    constexpr int UV = VEC * Storage<DT>::UNITS;  // 16-bit units per vector
    constexpr bool FLAT = READS == MergeReads::Dense;
    const uint32_t first = blockIdx.x * (THREADS * UNROLL);
    const uint32_t base = first + threadIdx.x;
    const int64_t flat0 = static_cast<int64_t>(row0) * nvec.d;  // the launch's first vector in a dense tensor
    if constexpr (READS != MergeReads::Few) {
        const uint32_t count = min(static_cast<uint32_t>(THREADS * UNROLL), total_vecs - first);
        if constexpr (FLAT) {
            if (threadIdx.x == 0) {
                prefetch_l2_range(v_a + (flat0 + first) * UV, static_cast<int64_t>(count) * UV * 2);
                prefetch_l2_range(v_b + (flat0 + first) * UV, static_cast<int64_t>(count) * UV * 2);
            }
        } else {
            const uint32_t lrow = nvec.div(first) + threadIdx.x;
            if (lrow <= nvec.div(first + count - 1)) {
                const uint32_t row = row0 + lrow, t = heads.div(row), h = row - t * heads.d;
                const int64_t bytes = static_cast<int64_t>(nvec.d) * UV * 2;
                prefetch_l2_range(v_a + (t * st.va_t + h * st.va_h), bytes);
                prefetch_l2_range(v_b + (t * st.vb_t + h * st.vb_h), bytes);
            }
        }
    }
    grid_dependency_wait();
    grid_launch_dependents();
    Pack<UV> a[UNROLL], b[UNROLL];
    float sa[UNROLL], sb[UNROLL];
    struct Place {
        uint32_t v, t, h;
        int64_t col;
    };
    auto place = [&](int j) {
        Place p;
        p.v = base + j * THREADS;
        const uint32_t lrow = nvec.div(p.v);
        const uint32_t row = row0 + lrow;  // rows of this launch start at row0
        p.t = heads.div(row);
        p.h = row - p.t * heads.d;
        p.col = static_cast<int64_t>(p.v - lrow * nvec.d) * UV;
        return p;
    };
    auto fetch = [&](int j, const Place &p) {
        a[j] = load<UV, Ld::Stream>(v_a + (FLAT ? (flat0 + p.v) * UV : p.t * st.va_t + p.h * st.va_h + p.col));
        b[j] = load<UV, Ld::Stream>(v_b + (FLAT ? (flat0 + p.v) * UV : p.t * st.vb_t + p.h * st.vb_h + p.col));
        sa[j] = lse_a[p.t * st.sa_t + p.h * st.sa_h];
        sb[j] = lse_b[p.t * st.sb_t + p.h * st.sb_h];
    };
    auto finish = [&](int j, const Place &p) {
        const MergeWeights mw = merge_weights(sa[j], sb[j]);
        store<UV, St::Stream>(v_out + (FLAT ? (flat0 + p.v) * UV : p.t * st.vo_t + p.h * st.vo_h + p.col),
                              merge_packs<DT, UV>(mw, a[j], b[j]));
        if (lse_out != nullptr && p.col == 0) lse_out[p.t * st.so_t + p.h * st.so_h] = mw.lse;
    };
    if constexpr (READS == MergeReads::Few) {
#pragma unroll
        for (int j = 0; j < UNROLL; ++j) {
            if (base + j * THREADS < total_vecs) {
                const Place p = place(j);
                fetch(j, p);
                finish(j, p);
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < UNROLL; ++j)
            if (base + j * THREADS < total_vecs) fetch(j, place(j));
#pragma unroll
        for (int j = 0; j < UNROLL; ++j)
            if (base + j * THREADS < total_vecs) finish(j, place(j));
    }
}

}  // namespace astra
