"""Rows that start at any element: the kernels for odd widths and pitches against the oracle, at the edges
of their ranges, every storage type, operand offsets of every alignment class, pitches that move the
operands against one another."""
import pytest
import torch

import oracle
import paper_2509_07506_b200 as astra
from paper_2509_07506_b200 import workloads as wl
from parity import check_values
from test_gpu_parity import f64, run_silu
from test_gpu_strided import pitched, untouched

pytestmark = pytest.mark.gpu

BF16, FP16, FP32 = wl.BF16, wl.FP16, wl.FP32


@pytest.mark.parametrize("dtype", [BF16, FP16, FP32])
@pytest.mark.parametrize("offset", [0, 1, 6])
@pytest.mark.parametrize("T,D", [(1, 511), (1, 513), (2, 515), (3, 1537), (7, 1538), (5, 2049), (33, 4099), (9, 14337),
                                 (40, 11012)])
def test_silu_ragged_rows(T, D, offset, dtype):
    run_silu(wl.silu_inputs(T, D, dtype, std=2.0, seed=D + offset), offset=offset)


@pytest.mark.parametrize("D,pitches", [(1001, (1001, 1003, 1008)), (1003, (1004, 1010, 1006)), (4099, (4104, 4104, 4104))])
def test_silu_ragged_pitches(D, pitches):
    """Output, gate and up that start differently in every row, and odd widths in aligned rows."""
    T, (po, pg, pu) = 21, pitches
    inp = wl.silu_inputs(T, D, BF16, std=2.0, seed=D)
    gb, gv = pitched(inp.input[:, :D].contiguous(), pg, 0)
    ub, uv = pitched(inp.input[:, D:].contiguous(), pu, 0)
    ob, ov = pitched(torch.zeros((T, D), dtype=torch.bfloat16), po, 0)
    astra.astra_silu_and_mul_ex(ov, gv, uv)
    check_values(f64(ov.cpu()), oracle.silu_and_mul(wl.bits(inp.input), BF16), BF16, what="silu ragged pitches")
    for buf in (gb, ub, ob):
        assert untouched(buf, 0, D)
