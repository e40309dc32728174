"""Rows that start at any element: the kernels for odd widths and pitches against the oracle, at the edges
of their ranges, every storage type, operand offsets of every alignment class, pitches that move the
operands against one another."""
import numpy as np
import pytest
import torch

import oracle
import paper_2509_07506_b200 as astra
from paper_2509_07506_b200 import workloads as wl
from parity import check_values
from test_gpu_allreduce import run_allreduce
from test_gpu_parity import f64, run_rmsnorm, run_silu
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


@pytest.mark.parametrize("dtype", [BF16, FP16, FP32])
@pytest.mark.parametrize("offset", [0, 1, 6, 15])
@pytest.mark.parametrize("T,H", [(1, 1025), (3, 1039), (17, 2051), (5, 5121), (4, 5135), (300, 4099), (6, 5137), (3, 8191),
                                 (7, 11007), (5, 16383), (3, 16401), (1030, 2050)])
def test_rmsnorm_ragged_rows(T, H, offset, dtype):
    run_rmsnorm(wl.rmsnorm_inputs(T, H, dtype, eps=1e-5, seed=H + offset), offset=offset)


@pytest.mark.parametrize("dtype", [BF16, FP16])
@pytest.mark.parametrize("T,H,weight_row", [(4000, 1025, 7), (4000, 1030, 1), (4000, 1038, 3), (3109, 1025, 11), (1500, 2051, 5),
                                            (1030, 4101, 2)])
def test_rmsnorm_ragged_rows_with_a_weight_of_their_own(T, H, weight_row, dtype):
    """The weight as a row of a wider [L, H] tensor, which starts at another place within 32 bytes than the first
    row, at the row counts where two vectors per thread make one wave."""
    run_rmsnorm(wl.rmsnorm_inputs(T, H, dtype, eps=1e-5, seed=T + H), weight_offset=weight_row * H)


@pytest.mark.parametrize("pads", [(0, 0, 0, 0), (16, 128, 0, 32), (16, 8, 0, 0)])
def test_rmsnorm_ragged_pitches(pads):
    """Pitches that keep the four tensors together modulo 32 bytes, and (last) pitches that do not."""
    T, H = 19, 4099
    inp = wl.rmsnorm_inputs(T, H, FP16, eps=1e-5, seed=sum(pads))
    (xb, xv), (rb, rv) = pitched(inp.x, H + pads[0], 0), pitched(inp.residual, H + pads[1], 0)
    (yb, yv), (ob, ov) = (pitched(torch.zeros_like(inp.x), H + p, 0) for p in pads[2:])
    astra.astra_fused_add_rmsnorm_ex(yv, ov, xv, rv, inp.weight.cuda(), inp.eps)
    oy, orr = oracle.fused_add_rmsnorm(wl.bits(inp.x), wl.bits(inp.residual), wl.bits(inp.weight), inp.eps, FP16)
    assert np.array_equal(wl.bits(ov.cpu().contiguous()), orr)
    check_values(f64(yv.cpu()), oy, FP16, what="rmsnorm ragged pitches")
    for buf in (xb, rb, yb, ob):
        assert untouched(buf, 0, H)


@pytest.mark.parametrize("dtype", [BF16, FP16, FP32])
@pytest.mark.parametrize("n_parts", [2, 4, 9])
@pytest.mark.parametrize("T,H,offset", [(3, 2049, 0), (16, 4099, 1), (129, 2051, 6), (9, 8189, 15), (5, 16383, 0), (4, 1027, 3)])
def test_allreduce_rmsnorm_ragged_rows(n_parts, T, H, offset, dtype):
    run_allreduce(wl.allreduce_rmsnorm_inputs(T, H, n_parts, dtype, seed=H + n_parts), offset=offset)


@pytest.mark.parametrize("n_parts", [2, 8])
@pytest.mark.parametrize("T,H,dtype,offset", [(150, 10256, BF16, 0), (149, 11008, FP16, 0), (151, 14336, BF16, 0), (150, 14335, BF16, 0),
                                              (150, 5632, FP32, 0), (3, 8200, FP32, 0), (2, 16384, FP32, 0), (3, 16383, FP32, 2)])
def test_allreduce_rmsnorm_wide_rows(n_parts, T, H, dtype, offset):
    """Rows whose residual is requested last (10241 to 14336 units, more rows than SMs) and binary32 rows of
    more than 16384 units, aligned and not."""
    run_allreduce(wl.allreduce_rmsnorm_inputs(T, H, n_parts, dtype, seed=H + n_parts), offset=offset)


@pytest.mark.parametrize("T,H", [(65, 8200), (64, 8200), (66, 16384), (65, 11008)])
def test_rmsnorm_wide_aligned_fp32_rows(T, H):
    run_rmsnorm(wl.rmsnorm_inputs(T, H, FP32, eps=1e-5, seed=H + T))
