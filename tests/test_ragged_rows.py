"""Index arithmetic of the kernels for rows that start at any element, run on the host: the geometry
functions of the kernel headers and the launch rule are compiled into a small program that walks every
alignment of every operand, widths around multiples of the vector size, every block shape that the rule gives
them, and all threads, and checks that each unit of a row belongs to exactly one thread, that every access lies inside its tensor and is aligned to its size."""
import subprocess


from paper_2509_07506_b200 import build as astra_build

PROGRAM = r"""
#include <cstdio>
#include <set>
#include <utility>
#include <vector>
#include "fused_allreduce_add_rmsnorm.cuh"
#include "silu_and_mul.cuh"
using namespace astra;

static long failures = 0;
static void expect(bool ok, const char *what, long a, long b, long c, long d) {
    if (!ok && failures++ < 5) printf("%s: %ld %ld %ld %ld\n", what, a, b, c, d);
}
static const uint16_t *at_unit(long u) { return reinterpret_cast<const uint16_t *>(4096 + 2 * u); }

// Body and edge of one row, over all threads of a block of `threads` with `vpt` vectors each.
template <int UNITS> static void norm_row(long row, long weight, int units, int vpt, int threads) {
    std::vector<int> owner(units, 0);
    for (int t = 0; t < threads; ++t) {
        const RaggedRow g = ragged_row<UNITS>(at_unit(row), at_unit(weight), units, t);
        for (int i = 0; i < vpt; ++i) {
            const int v = t + i * threads;
            if (v >= g.nvec) continue;
            const int at = g.first + v * 16;
            expect((row + at) % 16 == 0 && (weight + at - g.shift) % 16 == 0, "alignment", row, weight, units, at);
            expect(at >= 0 && at + 16 <= units, "body", row, weight, units, at);
            expect(at - g.shift >= 0 && at - g.shift + (g.shift ? 32 : 16) <= units, "weight", row, weight, units, at);
            for (int k = 0; k < 16; ++k) ++owner[at + k];
        }
        if (g.edge >= 0) {
            expect(g.edge + UNITS <= units, "edge", row, weight, units, g.edge);
            for (int k = 0; k < UNITS; ++k) ++owner[g.edge + k];
        }
    }
    for (int u = 0; u < units; ++u) expect(owner[u] == 1, "covered once", row, weight, units, u);
}

// All granules of a [rows, D] call with pitched operands; the only memory is the pages (2048 units) with a part of a row.
template <int UNITS> static void silu_rows(long o0, long a0, long b0, int rows, int D, long po, long pa, long pb) {
    const uint16_t *gate = at_unit(a0), *up = at_unit(b0);
    const uint32_t end_rows = silu_ragged_end_rows(rows, gate, up, D, pa, pb);
    std::set<long> pages;
    for (int r = 0; r < rows; ++r)
        for (long row : {a0 + r * pa, b0 + r * pb})
            for (long page = row / 2048; page <= (row + D - 1) / 2048; ++page) pages.insert(page);
    auto exists = [&](long at, long n) { return pages.count(at / 2048) && pages.count((at + n - 1) / 2048); };
    const long first = a0 < b0 ? a0 : b0, last = (rows - 1) * (a0 < b0 ? pb : pa) + (a0 < b0 ? b0 : a0) + D;
    const bool packed = b0 == a0 + D && pa == pb;  // one tensor, otherwise two
    for (int r = 0; r < rows; ++r) {
        std::vector<int> owner(D, 0);
        const uint16_t *o = at_unit(o0 + r * po), *a = at_unit(a0 + r * pa), *b = at_unit(b0 + r * pb);
        for (int n = 0; n < (D + 14) / 8; ++n) {
            const RaggedGranule g = ragged_granule(o, a, b, n, D, r == 0 || static_cast<uint32_t>(r) >= end_rows);
            if (g.at >= D) continue;
            expect((o0 + r * po + g.at) % 8 == 0, "granule", r, D, g.at, 0);
            expect(g.shift_a % UNITS == 0 && g.shift_b % UNITS == 0 && g.at % UNITS == 0, "units", r, D, g.at, 0);
            if (g.whole) {
                const long la = a0 + r * pa + g.at - g.shift_a, lb = b0 + r * pb + g.at - g.shift_b;
                const int na = g.shift_a ? 16 : 8, nb = g.shift_b ? 16 : 8;
                expect(la % 8 == 0 && lb % 8 == 0, "aligned loads", r, D, g.at, 0);
                expect(exists(la, na) && exists(lb, nb), "pages", r, D, g.at, la);
                if (packed) expect(la >= first && lb >= first && la + na <= last && lb + nb <= last, "tensor", r, D, g.at, la);
                else expect(la >= a0 && la + na <= a0 + (rows - 1) * pa + D && lb >= b0 && lb + nb <= b0 + (rows - 1) * pb + D,
                            "tensors", r, D, g.at, la);
            }
            for (int k = 0; k < 8; ++k) if (g.at + k >= 0 && g.at + k < D) ++owner[g.at + k];
        }
        for (int u = 0; u < D; ++u) expect(owner[u] == 1, "covered once", r, D, u, owner[u]);
    }
}

int main() {
    // every shape that the launch rules of the two norms give a width at any row count
    std::set<int> widths = {1055, 1056, 1057, 2051, 4099, 5120, 5135, 5136, 8191, 16383, 16399, 16400, 32767, 32782};
    for (int units = 1024; units <= 1041; ++units) widths.insert(units);
    for (int units : widths)
        for (bool binary32 : {false, true}) {
            std::set<std::pair<int, int>> shapes;
            for (int T = 1; T <= 6000; ++T)
                for (int vec : {1, 2, 4, 8}) {
                    const RaggedShape sh = rmsnorm_ragged_shape(T, units, binary32, vec);
                    if (sh.vpt > 0) shapes.insert({sh.vpt, sh.threads});
                }
            for (int T : {1, 100, 129, 148, 150, 296, 300, 500, 4096})
                for (int n_parts : {1, 2, 4, 8}) {
                    const AllreduceShape sh = allreduce_wide_shape(T, units, n_parts, binary32, true);
                    if (sh.vpt > 0) shapes.insert({sh.vpt, sh.threads});
                }
            expect(binary32 || units >= 16400 || !shapes.empty(), "shape", units, 0, 0, 0);
            for (auto [vpt, threads] : shapes)
                for (long row = 0; row < 16; ++row)
                    for (long weight = 0; weight < 16; ++weight) {
                        if (!binary32) norm_row<1>(row, weight, units, vpt, threads);
                        else if (units % 2 == 0 && row % 2 == 0 && weight % 2 == 0) norm_row<2>(row, weight, units, vpt, threads);
                    }
        }
    for (int D : {512, 513, 514, 519, 520, 527})
        for (int rows : {1, 2, 3, 5})
            for (long o = 0; o < 8; ++o)
                for (long a = 0; a < 8; ++a) {
                    silu_rows<1>(o, a, a + D, rows, D, D, 2 * D, 2 * D);        // the packed form
                    silu_rows<1>(o, a, (5 * a + 3) % 8, rows, D, D + 3, D, D + 1);
                    silu_rows<1>(o, a, a + D, rows, D, D, 2 * D + 1000, 2 * D + 1000);
                    for (long pitch : {2048L, 4096L, 8192L, 8193L})  // rows that begin or end a page, pages without a row
                        for (long at : {0L, 2048L - D}) silu_rows<1>(o, at + a, at + (5 * a + 3) % 8, rows, D, D, pitch, pitch);
                    if (D % 2 == 0 && o % 2 == 0 && a % 2 == 0) silu_rows<2>(o, a, a + D, rows, D, D, 2 * D, 2 * D);
                }
    printf("%ld failures\n", failures);
    return failures != 0;
}
"""


def test_every_unit_of_a_ragged_row_has_one_owner_and_stays_inside(tmp_path):
    src = tmp_path / "ragged.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "ragged"
    subprocess.check_call([astra_build._nvcc(), "-std=c++17", "-O1", "-gencode", "arch=compute_100a,code=sm_100a",
                           "-I", astra_build.INCLUDE, "-I", astra_build.CSRC, "-o", str(exe), str(src)])
    done = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stdout
