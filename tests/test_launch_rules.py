"""The rules that choose between a kernel for rows that start anywhere (or one that asks for its inputs ahead of
time) and the plain forms, at sizes where one of the two was measured to be the slower: the rules are host
functions of the kernel headers, compiled into a small program."""
import subprocess

from paper_2509_07506_b200 import build as astra_build

PROGRAM = r"""
#include <cstdio>
#include "fused_allreduce_add_rmsnorm.cuh"
#include "merge_attn_states_lse.cuh"
#include "silu_and_mul.cuh"
using namespace astra;

static int failures = 0;
#define EXPECT(want, call) do { if ((call) != (want)) { ++failures; printf("%s is not %s\n", #call, #want); } } while (0)

static void allreduce() {
    // (rows, units, partials, binary32, units per access of the narrow form)
    EXPECT(true, allreduce_keeps_narrow(150, 1060, 8, false, 4));
    EXPECT(true, allreduce_keeps_narrow(150, 3076, 4, false, 4));
    EXPECT(true, allreduce_keeps_narrow(296, 3588, 8, false, 4));
    EXPECT(true, allreduce_keeps_narrow(800, 1060, 2, false, 4));
    EXPECT(true, allreduce_keeps_narrow(3000, 3588, 2, false, 4));
    EXPECT(true, allreduce_keeps_narrow(16, 4100, 8, false, 4));
    EXPECT(false, allreduce_keeps_narrow(150, 4100, 4, false, 4));
    EXPECT(false, allreduce_keeps_narrow(300, 2084, 8, false, 4));
    EXPECT(false, allreduce_keeps_narrow(1500, 5124, 4, false, 4));
    EXPECT(false, allreduce_keeps_narrow(16, 14332, 8, false, 4));
    EXPECT(true, allreduce_keeps_narrow(150, 1604, 2, true, 4));
    EXPECT(true, allreduce_keeps_narrow(150, 1204, 8, true, 4));
    EXPECT(true, allreduce_keeps_narrow(16, 9220, 4, true, 4));
    EXPECT(true, allreduce_keeps_narrow(1024, 16380, 4, true, 4));
    EXPECT(false, allreduce_keeps_narrow(150, 4100, 4, true, 4));
    EXPECT(false, allreduce_keeps_narrow(1500, 4100, 2, true, 4));
    EXPECT(false, allreduce_keeps_narrow(1024, 16388, 4, true, 4));
    for (int units : {1027, 4099, 16387})
        for (int T : {1, 150, 4096}) EXPECT(false, allreduce_keeps_narrow(T, units, 4, false, 1));
}

static bool norm_is_ragged(int64_t T, int64_t units, bool binary32, int vec) {
    return rmsnorm_ragged_shape(T, units, binary32, vec).vpt > 0;
}

static void norm() {
    EXPECT(false, norm_is_ragged(400, 1060, false, 4));
    EXPECT(false, norm_is_ragged(256, 3164, false, 4));
    EXPECT(false, norm_is_ragged(400, 4100, false, 4));
    EXPECT(false, norm_is_ragged(8, 16388, false, 4));
    EXPECT(false, norm_is_ragged(400, 1058, false, 2));
    EXPECT(false, norm_is_ragged(1500, 2084, false, 4));
    EXPECT(false, norm_is_ragged(400, 4100, true, 4));
    EXPECT(false, norm_is_ragged(128, 5124, true, 4));
    EXPECT(false, norm_is_ragged(16, 32768, true, 8));
    EXPECT(false, norm_is_ragged(160, 22016, true, 8));
    EXPECT(true, norm_is_ragged(8, 4100, false, 4));
    EXPECT(true, norm_is_ragged(600, 4100, false, 4));
    EXPECT(true, norm_is_ragged(450, 8196, false, 4));
    EXPECT(true, norm_is_ragged(16384, 4100, false, 4));
    EXPECT(true, norm_is_ragged(128, 16388, false, 4));
    EXPECT(true, norm_is_ragged(1000, 2050, false, 2));
    EXPECT(true, norm_is_ragged(1024, 32768, true, 8));
    EXPECT(true, norm_is_ragged(149, 32768, true, 8));
    for (int units : {1027, 4099, 16383})
        for (int T : {1, 150, 4096}) EXPECT(true, norm_is_ragged(T, units, false, 1));
}

static void merge() {
    // (blocks, rows per block, dense values)
    EXPECT(MergeReads::Few, merge_strided_reads(4, 32, false));     // fp32 [8, 32, 64]
    EXPECT(MergeReads::Few, merge_strided_reads(64, 32, false));    // bf16 [64, 32, 128]
    EXPECT(MergeReads::Few, merge_strided_reads(160, 64, false));   // bf16 [256, 40, 64]
    EXPECT(MergeReads::Few, merge_strided_reads(40, 16, false));    // bf16 [16, 40, 256]
    EXPECT(MergeReads::Few, merge_strided_reads(20, 32, true));     // bf16 [16, 40, 128]
    EXPECT(MergeReads::Rows, merge_strided_reads(1024, 32, false)); // bf16 [1024, 32, 128]
    EXPECT(MergeReads::Rows, merge_strided_reads(160, 8, false));   // fp32 [32, 40, 256]
    EXPECT(MergeReads::Dense, merge_strided_reads(64, 32, true));   // bf16 [64, 32, 128]
    EXPECT(MergeReads::Dense, merge_strided_reads(2560, 32, true)); // bf16 [2048, 40, 128]
}

static void silu() {
    // (rows, units, binary32, units per access of the flat form)
    EXPECT(false, silu_takes_ragged(1, 1028, false, 4));
    EXPECT(false, silu_takes_ragged(1, 1026, false, 2));
    EXPECT(false, silu_takes_ragged(16384, 516, false, 4));
    EXPECT(false, silu_takes_ragged(8192, 4100, false, 4));
    EXPECT(false, silu_takes_ragged(4, 14336, false, 8));
    EXPECT(true, silu_takes_ragged(1, 1538, false, 2));
    EXPECT(true, silu_takes_ragged(1, 3076, true, 4));
    EXPECT(true, silu_takes_ragged(4, 1028, false, 4));
    EXPECT(true, silu_takes_ragged(1, 515, false, 1));
    EXPECT(true, silu_takes_ragged(8192, 8196, true, 4));
}

static void largest() {  // the widest rows and the most of them that the entry points accept
    for (int64_t units : {(1ll << 30) - 1, 1ll << 30, 700000003ll})
        for (int64_t T : {1ll, 1ll << 31, 1ll << 40})
            for (int vec : {1, 2, 4, 8})
                for (bool binary32 : {false, true}) {
                    EXPECT(false, norm_is_ragged(T, units, binary32, vec));
                    for (bool ragged : {false, true}) EXPECT(0, allreduce_wide_shape(T, units, 4, binary32, ragged).vpt);
                }
}

int main() {
    largest();
    allreduce();
    norm();
    merge();
    silu();
    return failures != 0;
}
"""


def test_rules_at_sizes_that_were_measured(tmp_path):
    src, exe = tmp_path / "rules.cu", tmp_path / "rules"
    src.write_text(PROGRAM)
    subprocess.check_call([astra_build._nvcc(), "-std=c++17", "-O1", "-gencode", "arch=compute_100a,code=sm_100a",
                           "-Xcompiler", "-fsanitize=undefined,-fno-sanitize-recover=all", "-I", astra_build.INCLUDE, "-I", astra_build.CSRC,
                           "-o", str(exe), str(src)])
    done = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert done.returncode == 0, done.stdout + done.stderr
