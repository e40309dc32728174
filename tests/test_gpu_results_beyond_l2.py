"""The size from which normalised rows and merged values are stored for nobody to find in L2, from both sides: the norm's
residual bit for bit and its rows, from all over the call, against the oracle; the merge against smaller calls."""
import numpy as np
import pytest
import torch

import oracle
import paper_2509_07506_b200 as astra
from paper_2509_07506_b200 import workloads as wl
from parity import check_values

pytestmark = pytest.mark.gpu
LINE = 56 << 20  # bytes of x
CODE = {torch.bfloat16: wl.BF16, torch.float16: wl.FP16, torch.float32: wl.FP32}


@pytest.mark.parametrize("dtype", list(CODE))
@pytest.mark.parametrize("H", [4096, 1040, 14336, 4100, 4099, 1025])
@pytest.mark.parametrize("beyond", [-1, 0, 3])
def test_rows(dtype, H, beyond):
    T = LINE // (torch.empty(0, dtype=dtype).element_size() * H) + beyond
    g = torch.Generator(device="cuda")
    g.manual_seed(H + beyond)
    mk = lambda *shape: torch.randn(shape, generator=g, device="cuda").to(dtype)  # noqa: E731
    x, r, w = mk(T, H), mk(T, H), mk(H)
    rows = sorted({*range(0, T, max(1, T // 61)), *range(T - 5, T)})
    some_x, some_r, want_r = x[rows].cpu(), r[rows].cpu(), (x.float() + r.float()).to(dtype)
    astra.astra_fused_add_rmsnorm(x, r, w, 1e-5)
    assert torch.equal(r.view(torch.uint8), want_r.view(torch.uint8))
    oy, orr = oracle.fused_add_rmsnorm(wl.bits(some_x), wl.bits(some_r), wl.bits(w.cpu()), 1e-5, CODE[dtype])
    assert np.array_equal(wl.bits(r[rows].cpu()), orr)
    check_values(x[rows].cpu().to(torch.float64).numpy(), oy, CODE[dtype], what="fused_add_rmsnorm")
    assert x.isfinite().all()


@pytest.mark.parametrize("dtype", list(CODE))
@pytest.mark.parametrize("heads,D", [(32, 128), (5, 80), (3, 16)])
@pytest.mark.parametrize("beyond", [-1, 0, 3])
def test_merged_values(dtype, heads, D, beyond):
    """Elementwise: one call against its two halves, which are below that size, bit for bit."""
    T = -(-LINE // (torch.empty(0, dtype=dtype).element_size() * heads * D)) + beyond
    g = torch.Generator(device="cuda")
    g.manual_seed(D + beyond)
    mk = lambda *shape: torch.randn(shape, generator=g, device="cuda")  # noqa: E731
    va, vb, sa, sb = mk(T, heads, D).to(dtype), mk(T, heads, D).to(dtype), mk(T, heads) * 8, mk(T, heads) * 8
    sa[T // 3:T // 3 + 2] = float("-inf")
    out, lse, want, want_lse = torch.empty_like(va), torch.empty_like(sa), torch.empty_like(va), torch.empty_like(sa)
    half = T // 2 // 32 * 32
    for at in (slice(0, half), slice(half, T)):
        astra.astra_merge_attn_states_lse(want[at], want_lse[at], va[at], sa[at], vb[at], sb[at])
    astra.astra_merge_attn_states_lse(out, lse, va, sa, vb, sb)
    assert torch.equal(out.view(torch.uint8), want.view(torch.uint8)) and torch.equal(lse, want_lse)
