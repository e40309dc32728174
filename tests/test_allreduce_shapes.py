"""The launch shapes of the all-reduce norm: the figures that the choice rests on against the compiler and the
device.  A small program instantiates the kernels of the shape tables; the compiler prints the registers it
gave them, the program the tables and, on a device, how many blocks of them an SM really holds."""
import re
import subprocess

import pytest

from paper_2509_07506_b200 import build as astra_build

PROGRAM = r"""
#include <cstdio>
#include <cuda_runtime.h>
#include "fused_allreduce_add_rmsnorm.cuh"
using namespace astra;

template <bool RAGGED, int I> const void *kernel() {
    constexpr WideShape sh = (RAGGED ? kRaggedShapes : kWideShapes)[STORAGE == ASTRA_FP32][I];
    if constexpr (RAGGED) return (const void *)fused_allreduce_add_rmsnorm_ragged_kernel<STORAGE, sh.vpt, sh.group, sh.late>;
    else return (const void *)fused_allreduce_add_rmsnorm_reg_kernel<STORAGE, 16 / Storage<STORAGE>::UNITS, sh.vpt, sh.group, false, sh.late>;
}

template <bool RAGGED, int I> void row(bool device) {
    constexpr WideShape sh = (RAGGED ? kRaggedShapes : kWideShapes)[STORAGE == ASTRA_FP32][I];
    const void *k = kernel<RAGGED, I>();
    printf("shape %d %d %d %d %d\n", RAGGED, sh.vpt, sh.group, sh.late, sh.regs);
    for (int threads = sh.min_threads; device && threads <= sh.max_threads; threads += 32) {
        int blocks = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k, threads, 0) != cudaSuccess) blocks = -1;
        printf("blocks %d %d %d\n", threads, resident_blocks(sh.regs, threads), blocks);
    }
}

int main(int argc, char **) {
    const bool device = argc > 1;
    row<false, 0>(device), row<false, 1>(device), row<false, 2>(device), row<false, 3>(device), row<false, 4>(device);
    row<true, 0>(device), row<true, 1>(device), row<true, 2>(device), row<true, 3>(device), row<true, 4>(device);
    return 0;
}
"""


@pytest.fixture(scope="module")
def programs(tmp_path_factory):
    """Storage type -> (program, {(ragged, vpt, group, late): registers}), as compiled."""
    dir, running = tmp_path_factory.mktemp("shapes"), {}
    (dir / "shapes.cu").write_text(PROGRAM)
    flags = [f for f in astra_build.NVCC_FLAGS if f not in ("-shared", "-Xcompiler", "-fPIC")]
    for dt in (0, 1, 2):
        cmd = [astra_build._nvcc(), *flags, f"-DSTORAGE={dt}", "-Xptxas", "-v", "-I", astra_build.INCLUDE, "-I", astra_build.CSRC,
               "-o", str(dir / f"shapes{dt}"), str(dir / "shapes.cu")]
        running[dt] = subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    built = {}
    for dt, proc in running.items():
        out, _ = proc.communicate(timeout=900)
        assert proc.returncode == 0, out[-2000:]
        registers = {}
        for name, regs in re.findall(r"Compiling entry function '(\w+)'.*?Used (\d+) registers", out, flags=re.S):
            value = [int(v) for v in re.findall(r"L[ib](\d+)E", name)]
            if "ragged" in name:      # <DT, VPT, GROUP, LATE_R>
                registers[(1, value[1], value[2], value[3])] = int(regs)
            elif "_reg_kernel" in name:  # <DT, VEC, VPT, GROUP, DENSE, LATE_R>
                registers[(0, value[2], value[3], value[5])] = int(regs)
        built[dt] = (str(dir / f"shapes{dt}"), registers)
    return built


def rows(program, *args):
    out = subprocess.run([program, *args], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    return [(line.split()[0], *map(int, line.split()[1:])) for line in out.stdout.splitlines()]


def test_tables_state_the_registers_that_the_compiler_gives(programs):
    """Allocated in eights, so that is what the tables hold."""
    for dt, (program, registers) in programs.items():
        told = {row[1:5]: row[5] for row in rows(program)}
        assert len(told) == 10
        assert told == {k: (registers[k] + 7) // 8 * 8 for k in told}, dt


@pytest.mark.gpu
def test_as_many_blocks_are_resident_as_the_choice_counts(programs):
    for dt, (program, _) in programs.items():
        counted = [row[1:] for row in rows(program, "device") if row[0] == "blocks"]
        assert len(counted) > 100
        assert [r for r in counted if r[1] != r[2]] == [], dt
