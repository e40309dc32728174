// Runs of calls of one kind and shape (call_runs.h): which of them share a launch, and the launches.
// Same conventions as the entry points: nothing is allocated, kept or waited for.
#include <cuda_runtime.h>

#include "astra.h"
#include "call_runs.cuh"
#include "call_runs.h"
#include "fastcall.h"
#include "launch.cuh"

namespace {

using namespace astra;
using namespace astra::host;

struct Range {
    const void *at;
    int64_t bytes;
    bool meets(const Range &o) const { return bytes > 0 && o.bytes > 0 && overlaps(at, bytes, o.at, o.bytes); }
    bool same(const Range &o) const { return at == o.at && bytes == o.bytes; }
};

// What a call reads and writes, and how wide its accesses are.  usable: the operands are such that the entry
// point accepts the call and a run's kernel can take it.
struct Footprint {
    Range read[4], written[2];
    int reads = 0, writes = 0, vec = 0;
    bool usable = false;
};

struct Shape {
    int kind;
    int64_t ext[3];
    float eps;
    astra_dtype_t dtype;
    int64_t units() const { return units_per_elem(dtype); }
    int64_t extents() const { return kind == KIND_MERGE ? 3 : 2; }
};

Footprint footprint(const Shape &sh, const astra_run_call &c) {
    Footprint f;
    void *const *p = c.ptr;
    const int64_t elem = 2 * sh.units(), a = sh.ext[0], b = sh.ext[1];
    VecPick pick(16);
    if (sh.kind == KIND_RMSNORM) {  // x, residual, weight
        f.read[0] = {p[2], b * elem};
        f.written[0] = {p[0], a * b * elem};
        f.written[1] = {p[1], a * b * elem};
        f.reads = 1, f.writes = 2;
        pick.extent(b * sh.units()).pointer(p[0]).pointer(p[1]).pointer(p[2]);
        f.usable = p[0] && p[1] && p[2] && !f.written[0].meets(f.written[1]) && !f.read[0].meets(f.written[0]) &&
                   !f.read[0].meets(f.written[1]) && norm_run_shape(a, b * sh.units(), pick.vec).threads != 0;
    } else if (sh.kind == KIND_SILU) {  // out, input
        f.read[0] = {p[1], 2 * a * b * elem};
        f.written[0] = {p[0], a * b * elem};
        f.reads = f.writes = 1;
        pick.extent(b * sh.units()).pointer(p[0]).pointer(p[1]);
        f.usable = p[0] && p[1] && !f.read[0].meets(f.written[0]) && pick.vec >= 8;
    } else {  // v_out, lse_out, v_a, lse_a, v_b, lse_b
        const int64_t values = a * b * sh.ext[2] * elem, scores = a * b * 4;
        f.written[0] = {p[0], values};
        f.written[1] = {p[1], p[1] ? scores : 0};
        f.read[0] = {p[2], values};
        f.read[1] = {p[3], scores};
        f.read[2] = {p[4], values};
        f.read[3] = {p[5], scores};
        f.reads = 4, f.writes = 2;
        pick.extent(sh.ext[2] * sh.units()).pointer(p[0]).pointer(p[2]).pointer(p[4]);
        bool ok = p[0] && p[2] && p[3] && p[4] && p[5] && aligned(p[1], 4) && aligned(p[3], 4) && aligned(p[5], 4);
        ok = ok && !f.written[0].meets(f.written[1]);
        for (int r = 0; r < 4; ++r) {
            const bool in_place = (r == 0 || r == 2) && f.read[r].same(f.written[0]);
            ok = ok && (in_place || !f.read[r].meets(f.written[0])) && !f.read[r].meets(f.written[1]);
        }
        f.usable = ok && pick.vec >= 8;
    }
    f.vec = pick.vec;
    return f;
}

// May calls p and q share a launch?  Neither reads what the other writes, and what both write is the same tensor
// or two that do not meet.  The norm's residual is read and written by each call's own threads in order: it has
// to be one and the same tensor, and the hidden states two.
bool together(const Shape &sh, const Footprint &p, const Footprint &q) {
    const bool norm = sh.kind == KIND_RMSNORM;
    if (norm && (p.vec != q.vec || !p.written[1].same(q.written[1]))) return false;
    for (int w = 0; w < p.writes; ++w)
        for (int r = 0; r < q.reads; ++r)
            if (p.written[w].meets(q.read[r])) return false;
    for (int w = 0; w < q.writes; ++w)
        for (int r = 0; r < p.reads; ++r)
            if (q.written[w].meets(p.read[r])) return false;
    for (int w = 0; w < p.writes; ++w)
        for (int v = 0; v < q.writes; ++v)
            if (p.written[w].meets(q.written[v]) && !(w == v && p.written[w].same(q.written[v]) && !(norm && w == 0))) return false;
    return true;
}

// Do the sizes allow a run at all?  (One launch, 31-bit vector indices, and nothing that overflows here.)
bool runnable(const Shape &sh) {
    if (!valid_dtype(sh.dtype)) return false;
    int64_t total = sh.units();
    for (int i = 0; i < sh.extents(); ++i) {
        if (sh.ext[i] <= 0 || sh.ext[i] > (1ll << 33) / total) return false;
        total *= sh.ext[i];
    }
    return total / 8 <= kMaxVecsPerLaunch && (sh.kind != KIND_RMSNORM || sh.ext[0] <= kMaxRowsPerLaunch / 8);
}

// Is a launch of `count` calls the faster?  The elementwise kernels of a run keep fewer threads resident than those of
// single calls (96 registers silu, 104 to 116 merge) and lose where a single call fills the GPU: us a call together / one by one, silu
// 2.05 / 3.33 at [256, 14336] but 31 / 26 for two calls at [2048, 14336]; merge 1.92 / 2.50 at [256, 64, 128] but 3.45 / 3.14
// at [512, 64, 128].  Norms, which keep their residual, gain at every size (24 / 41 us at [8192, 4096], 8 calls).  Two or
// three calls have too few loads in flight beyond smaller sizes (silu 5.1 / 4.1 at [256, 14336], merge 4.1 / 3.1 at
// [256, 64, 128], norm 20 / 16 at [4096, 4096], 3.1 / 3.1 at [256, 4096]).
bool worth(const Shape &sh, int count) {
    int64_t units = sh.units();
    for (int i = 0; i < sh.extents(); ++i) units *= sh.ext[i];
    if (count < 4) return count > 1 && units <= (sh.kind == KIND_RMSNORM ? 1 << 22 : sh.kind == KIND_SILU ? 1 << 21 : 1 << 20);
    return sh.kind == KIND_RMSNORM || units <= (sh.kind == KIND_SILU ? 1 << 22 : 1 << 21);
}

astra_status_t issue_one(const Shape &sh, const astra_run_call &c, void *stream) {
    void *const *p = c.ptr;
    switch (sh.kind) {
        case KIND_RMSNORM: return astra_fused_add_rmsnorm(p[0], p[1], p[2], sh.ext[0], sh.ext[1], sh.eps, sh.dtype, stream);
        case KIND_SILU: return astra_silu_and_mul(p[0], p[1], sh.ext[0], sh.ext[1], sh.dtype, stream);
        default:
            return astra_merge_attn_states_lse(p[0], static_cast<float *>(p[1]), p[2], static_cast<const float *>(p[3]), p[4],
                                               static_cast<const float *>(p[5]), sh.ext[0], sh.ext[1], sh.ext[2], sh.dtype,
                                               stream);
    }
}

template <int DT> cudaError_t launch_norms(const Shape &sh, const astra_run_call *c, int n, int vec, cudaStream_t stream) {
    constexpr int U = Storage<DT>::UNITS;
    const NormRunShape f = norm_run_shape(sh.ext[0], sh.ext[1] * U, vec);
    RmsnormRun run = {};
    for (int i = 0; i < n; ++i) {
        run.x[i] = static_cast<uint16_t *>(c[i].ptr[0]);
        run.w[i] = static_cast<const uint16_t *>(c[i].ptr[2]);
    }
    run.r = static_cast<uint16_t *>(c[0].ptr[1]);
    run.n = n;
    run.H = static_cast<int>(sh.ext[1]);
    run.blocks = f.blocks;
    run.eps = sh.eps;
    run.inv_H = 1.0f / static_cast<float>(run.H);
    const unsigned grid = static_cast<unsigned>(sh.ext[0] * f.blocks);
    if (f.blocks > 1)
        return launch_clustered(fused_add_rmsnorm_run_kernel<DT, 8 / U, 8, 256, true>, grid, f.threads, f.blocks, stream, run);
    if (f.uvec == 8) return launch(fused_add_rmsnorm_run_kernel<DT, 8 / U, 2, 512, false>, grid, f.threads, stream, run);
    return launch(fused_add_rmsnorm_run_kernel<DT, 16 / U, 2, 512, false>, grid, f.threads, stream, run);
}

template <int DT> cudaError_t launch_silus(const Shape &sh, const astra_run_call *c, int n, cudaStream_t stream) {
    SiluRun run = {};
    for (int i = 0; i < n; ++i) {
        run.out[i] = static_cast<uint16_t *>(c[i].ptr[0]);
        run.in[i] = static_cast<const uint16_t *>(c[i].ptr[1]);
    }
    run.n = n;
    run.D = sh.ext[1] * sh.units();
    run.nvec = FastDiv::make(static_cast<uint32_t>(run.D / 8));
    run.total_vecs = static_cast<uint32_t>(sh.ext[0] * (run.D / 8));
    return launch(silu_and_mul_run_kernel<DT>, (run.total_vecs + kRunThreads - 1) / kRunThreads, kRunThreads, stream, run);
}

template <int DT> cudaError_t launch_merges(const Shape &sh, const astra_run_call *c, int n, cudaStream_t stream) {
    MergeRun run = {};
    for (int i = 0; i < n; ++i) {
        run.v_out[i] = static_cast<uint16_t *>(c[i].ptr[0]);
        run.lse_out[i] = static_cast<float *>(c[i].ptr[1]);
        run.v_a[i] = static_cast<const uint16_t *>(c[i].ptr[2]);
        run.lse_a[i] = static_cast<const float *>(c[i].ptr[3]);
        run.v_b[i] = static_cast<const uint16_t *>(c[i].ptr[4]);
        run.lse_b[i] = static_cast<const float *>(c[i].ptr[5]);
    }
    run.n = n;
    const int64_t nvec = sh.ext[2] * sh.units() / 8;
    run.nvec = FastDiv::make(static_cast<uint32_t>(nvec));
    run.total_vecs = static_cast<uint32_t>(sh.ext[0] * sh.ext[1] * nvec);
    return launch(merge_attn_states_lse_run_kernel<DT>, (run.total_vecs + kRunThreads - 1) / kRunThreads, kRunThreads, stream, run);
}

astra_status_t issue_together(const Shape &sh, const astra_run_call *c, int n, int vec, cudaStream_t stream) {
    cudaError_t err = cudaSuccess;
    if (sh.kind == KIND_RMSNORM) ASTRA_FOR_DTYPE(sh.dtype, err = launch_norms<DT>(sh, c, n, vec, stream));
    else if (sh.kind == KIND_SILU) ASTRA_FOR_DTYPE(sh.dtype, err = launch_silus<DT>(sh, c, n, stream));
    else ASTRA_FOR_DTYPE(sh.dtype, err = launch_merges<DT>(sh, c, n, stream));
    return launch_status(err);
}

// How many of the n calls, from the first on, share a launch; vec is the width of its accesses.
int calls_together(const Shape &sh, const astra_run_call *calls, int32_t n, int *vec) {
    Footprint f[kMaxRun];
    f[0] = footprint(sh, calls[0]);
    *vec = f[0].vec;
    int count = 1;
    bool more = f[0].usable;
    while (more && count < kMaxRun && count < n) {
        f[count] = footprint(sh, calls[count]);
        more = f[count].usable;
        for (int k = 0; more && k < count; ++k) more = together(sh, f[k], f[count]);
        count += more;
    }
    return worth(sh, count) ? count : 1;
}

// The calls of each launch, in order, to issue(first call, count, vec); stops at what is not ASTRA_OK.
template <typename ISSUE>
astra_status_t for_each_launch(int kind, int32_t n, const astra_run_call *calls, const int64_t *ext, float eps, astra_dtype_t dtype,
                               ISSUE issue) {
    if ((kind != KIND_RMSNORM && kind != KIND_SILU && kind != KIND_MERGE) || n < 0) return ASTRA_ERR_BAD_SHAPE;
    if (n == 0) return ASTRA_OK;
    if (!calls || !ext) return ASTRA_ERR_NULL_POINTER;
    const Shape sh = {kind, {ext[0], ext[1], kind == KIND_MERGE ? ext[2] : 0}, eps, dtype};
    const bool may_run = runnable(sh);
    for (int32_t i = 0; i < n;) {
        int vec = 0;
        const int count = may_run ? calls_together(sh, calls + i, n - i, &vec) : 1;
        const astra_status_t st = issue(sh, calls + i, count, vec);
        if (st != ASTRA_OK) return st;
        i += count;
    }
    return ASTRA_OK;
}

}  // namespace

extern "C" astra_status_t astra_issue_run(int kind, int32_t n, const astra_run_call *calls, const int64_t *ext, float eps,
                                          astra_dtype_t dtype, void *cuda_stream) {
    return for_each_launch(kind, n, calls, ext, eps, dtype, [&](const Shape &sh, const astra_run_call *c, int count, int vec) {
        return count > 1 ? issue_together(sh, c, count, vec, static_cast<cudaStream_t>(cuda_stream)) : issue_one(sh, *c, cuda_stream);
    });
}

extern "C" astra_status_t astra_plan_run(int kind, int32_t n, const astra_run_call *calls, const int64_t *ext, astra_dtype_t dtype,
                                         int32_t *counts, int32_t *launches) {
    if (!counts || !launches) return ASTRA_ERR_NULL_POINTER;
    *launches = 0;
    return for_each_launch(kind, n, calls, ext, 0.0f, dtype, [&](const Shape &, const astra_run_call *, int count, int) {
        counts[(*launches)++] = count;
        return ASTRA_OK;
    });
}
