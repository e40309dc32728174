"""silu_and_mul: which form of the sigmoid a warp takes is decided by its lanes together, and what an element becomes by
itself alone.  Rows with and without gates below -40 in some places have the same bits in all others, in each
kernel (flat with 2- to 32-byte vectors, ragged rows, runs of captured calls)."""
import pytest
import torch

import paper_2509_07506_b200 as astra

pytestmark = pytest.mark.gpu
BITS = {torch.bfloat16: torch.int16, torch.float16: torch.int16, torch.float32: torch.int32}


def outputs(inputs, way):
    outs = [torch.empty(t.shape[0], t.shape[1] // 2, dtype=t.dtype, device="cuda") for t in inputs]
    if way == "run":
        astra.CapturedCalls([astra.prepare_silu_and_mul(o, t) for o, t in zip(outs, inputs)]).replay()
    else:
        for o, t in zip(outs, inputs):
            astra.astra_silu_and_mul(o, t)
    torch.cuda.synchronize()
    return outs


@pytest.mark.parametrize("dtype", list(BITS))
@pytest.mark.parametrize("T,D,way", [(1, 1, "direct"), (3, 2, "direct"), (5, 36, "direct"), (16, 4096, "direct"), (300, 14336, "direct"),
                                     (9, 1037, "direct"), (9, 4099, "direct"), (16, 4096, "run"), (3, 1000, "run")])
def test_far_gates_change_nothing_beside_them(dtype, T, D, way):
    g = torch.Generator().manual_seed(T + D)
    plain = torch.randn(T, 2 * D, generator=g) * 6
    far = plain.clone()
    at = torch.arange(T * D).view(T, D)
    moved = (at * 11 + at // 7) % 41 == 0   # a few lanes of most warps, and every lane of none
    far[:, :D][moved] = -40.0 - 100 * torch.rand(int(moved.sum()), generator=g)
    alone = torch.where(moved, far[:, :D], -50.0)  # the same far gates among others, the rest of the gates far as well
    alone = torch.cat([alone, plain[:, D:]], 1)
    p, f, a = (o.view(BITS[dtype]).cpu() for o in outputs([t.to(dtype).cuda() for t in (plain, far, alone)], way))
    assert torch.equal(p[~moved], f[~moved])
    assert torch.equal(f[moved], a[moved])
