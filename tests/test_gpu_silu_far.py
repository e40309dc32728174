"""silu_and_mul around the gate value (-40) below which the sigmoid takes its overflow-free form: every position of a
vector, next to ordinary values, at every alignment, against the oracle; and the same elements give the same bits
however their rows are cut into vectors."""
import numpy as np
import pytest
import torch

import oracle
import paper_2509_07506_b200 as astra
from paper_2509_07506_b200 import workloads as wl
from parity import check_values, ulp

FAR = [-39.5, -39.99, -40.0, -40.01, -40.25, -60.0, -80.0, -87.3, -88.0, -95.0, -103.9, -104.0, -150.0, -173.0, -180.0, -1000.0,
       -0.0, 0.0, 88.0, 104.0, 3.0, -3.0]


def operands(T, D, dtype):
    g = torch.Generator().manual_seed(T + D)
    a, b = torch.randn(T, D, generator=g) * 3, torch.randn(T, D, generator=g) * 50
    at = torch.arange(T * D)
    pick = (at * 7 + at // 16) % 13 == 0  # wanders over all positions of 8- and 16-unit vectors
    a.view(-1)[pick] = torch.tensor(FAR).repeat(-(-int(pick.sum()) // len(FAR)))[:int(pick.sum())]
    return a.to(dtype), b.to(dtype)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16, torch.float32])
@pytest.mark.parametrize("T,D", [(1, 8), (3, 40), (5, 1037), (4, 4096), (300, 14336), (9, 4099), (2, 1028)])
def test_far_elements(dtype, T, D):
    a, b = operands(T, D, dtype)
    results = []
    for offset in (0, 1, 2, 8):
        buf = torch.zeros(offset + 2 * T * D, dtype=dtype, device="cuda")
        inp = buf[offset:].view(T, 2 * D)
        inp.copy_(torch.cat([a, b], 1))
        out = torch.empty(offset + T * D, dtype=dtype, device="cuda")[offset:].view(T, D)
        astra.astra_silu_and_mul(out, inp)
        results.append(out.cpu())
    code = {torch.bfloat16: wl.BF16, torch.float16: wl.FP16, torch.float32: wl.FP32}[dtype]
    want = oracle.silu_and_mul(wl.bits(torch.cat([a, b], 1).contiguous()), code)
    for r in results[1:]:
        assert np.array_equal(wl.bits(r.contiguous()), wl.bits(results[0].contiguous()))
    # e^a is a binary32 number, whose smallest step is 2^-149: below 2^-126 it is off by half a step (and the factor
    # 1 / (1 + e^a), which is 1 there, by none), so the result by |a b| 2^-150, taken twice for its own rounding.
    # binary32: the exponent's argument is rounded, too, which costs 2 |a| ulp besides the gate's 16.
    extra = (a.double() * b.double()).abs().numpy() * 2.0 ** -149
    if dtype == torch.float32:
        extra = extra + 2 * a.abs().double().numpy() * ulp(want, code)
    check_values(results[0].double().numpy(), want, code, extra=extra, what="silu")


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16, torch.float32])
def test_values_that_are_not_finite(dtype):
    inf, nan = float("inf"), float("nan")
    a = torch.tensor([inf, -inf, nan, -nan, -41.0, -41.0, -90.0, 1.0] * 4).to(dtype)
    b = torch.tensor([2.0, 2.0, 1.0, 1.0, inf, nan, -inf, -inf] * 4).to(dtype)
    inp = torch.cat([a, b]).view(1, -1).cuda()
    out = torch.empty(1, a.numel(), dtype=dtype, device="cuda")
    astra.astra_silu_and_mul(out, inp)
    got = out.cpu().float().view(-1, 8)
    for row in got:
        assert row[0] == inf and row[1:4].isnan().all() and row[4] == -inf and row[5].isnan() and row[6] == inf and row[7] == -inf
