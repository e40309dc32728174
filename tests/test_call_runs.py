"""Calls that are captured together: one launch for several calls of one kind against the same calls issued one by one,
at the edges of the forms (rows per cluster, calls per exchange and per launch, widths) and for operands that are shared
between calls in every way that allows a common launch or forbids it."""
import pytest
import torch

import paper_2509_07506_b200 as astra
from paper_2509_07506_b200 import binding, graphs

A = 1 << 20
BITS = {torch.bfloat16: torch.int16, torch.float16: torch.int16, torch.float32: torch.int32}


def prepared(kind, ranges, ext, eps=0.0, dtype=0, parts=()):
    ready = binding._fast.prepare(kind, ranges, ext, eps, dtype, parts)
    return binding.PreparedCall("call", None, None, torch.device("cuda", 0), (), ready)


def test_like_calls_of_a_group_form_runs(monkeypatch):
    binding.load_library()
    fast = binding._fast
    monkeypatch.setattr(graphs, "_pointer_attributes", lambda: None)
    monkeypatch.setattr(fast, "one_address_each", lambda calls, query: True)
    norm = lambda x, r, H=64, eps=1e-6: prepared(fast.KIND_RMSNORM, (A * x, A * r, A * 99), (4, H), eps)  # noqa: E731
    silu = lambda o, i: prepared(fast.KIND_SILU, (A * o, A * i), (4, 64))  # noqa: E731
    # one residual and one output: two groups, each a run; in the order given on request
    calls = [norm(1, 2), silu(10, 11), norm(3, 2), silu(10, 12), norm(4, 2)]
    assert graphs._plan(calls, 2) == [(0, [calls[0], calls[2], calls[4]]), (1, [calls[1], calls[3]])]
    assert graphs._plan(calls, 1) == [(0, [c]) for c in calls]
    # an activation that reads a norm's result comes between the norms
    calls = [norm(1, 2), silu(10, 1), norm(3, 2)]
    assert [run for _, run in graphs._plan(calls, 2)] == [[c] for c in calls]
    # another width or epsilon, or the all-reduce form, is another run
    for other in (norm(3, 2, 32), norm(3, 2, 64, 1e-5),
                  prepared(fast.KIND_ALLREDUCE_RMSNORM, (A * 3, A * 2, A * 99), (4, 64), 1e-6, 0, (A * 5,))):
        calls = [norm(1, 2), other]
        assert [run for _, run in graphs._plan(calls, 2)] == [[c] for c in calls]


def test_runs_are_refused_unless_the_calls_are_alike():
    binding.load_library()
    fast = binding._fast
    a = fast.prepare(fast.KIND_SILU, (A, 2 * A), (4, 64), 0.0, 0, ())
    b = fast.prepare(fast.KIND_SILU, (A, 2 * A), (4, 32), 0.0, 0, ())
    for calls in ([], [a, b], [a, None], [None, a]):
        with pytest.raises(ValueError):
            fast.launch_run(calls, 0)
    with pytest.raises(TypeError):
        fast.launch_run((a,), 0)
    # a call that the entry point refuses ends the run with its status, launching nothing
    overlapping = fast.prepare(fast.KIND_SILU, (A, A), (4, 64), 0.0, 0, ())
    assert fast.launch_run([overlapping, a], 0) == binding.ASTRA_ERR_OVERLAP
    misaligned = fast.prepare(fast.KIND_RMSNORM, (A + 1, 2 * A, 3 * A), (4, 64), 1e-6, 0, ())
    assert fast.launch_run([misaligned, misaligned], 0) == binding.ASTRA_ERR_MISALIGNED
    empty = fast.prepare(fast.KIND_SILU, (0, 0), (0, 64), 0.0, 0, ())
    assert fast.launch_run([empty, empty], 0) == binding.ASTRA_OK


def in_order(t):
    """The bit patterns as integers in the order of the values."""
    b = t.view(BITS[t.dtype]).long()
    return torch.where(b < 0, -(1 << (8 * t.element_size() - 1)) - b, b)


def compare(build, ulps=0, passes=2):
    """build() -> (calls, tensors, indexes of those that may differ by `ulps`): replays against the calls in order."""
    calls, got, near = build()
    start = [t.clone() for t in got]
    graph = astra.CapturedCalls(calls)
    for t, s in zip(got, start):
        t.copy_(s)
    ref_calls, want, _ = build()
    for _ in range(passes):
        graph.replay()
        for call in ref_calls:
            call()
    torch.cuda.synchronize()
    for i, (p, q) in enumerate(zip(got, want)):
        assert not p.isnan().any(), i
        if i in near:
            assert (in_order(p) - in_order(q)).abs().max() <= ulps, i
        else:
            assert torch.equal(p.view(BITS[p.dtype]), q.view(BITS[q.dtype])), i


def maker(seed, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return lambda *shape, dt=dtype: torch.randn(shape, generator=g, device="cuda").to(dt)


# The squares of a row are summed in another order than by a single call, so rstd differs by a few 2^-24: y is the same
# or the neighbouring value of a 16-bit type, and within 16 ulp (the gate of the other binary32 tests) for binary32.
@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16, torch.float32])
@pytest.mark.parametrize("T,H,n", [(1, 4096, 64), (3, 256, 2), (16, 2048, 7), (37, 4096, 8), (38, 4096, 9), (37, 2056, 15), (16, 8192, 17),
                                   (74, 2056, 16), (75, 4096, 5), (75, 8192, 4), (100, 520, 65), (130, 4104, 3), (300, 1032, 130),
                                   (16, 8200, 4), (5, 4100, 4), (2, 4099, 3), (1, 8, 70)])
def test_norms_on_one_residual(dtype, T, H, n):
    def build():
        mk = maker(T + H + n, dtype)
        xs, r, ws = mk(n, T, H), mk(T, H), mk(n, H)
        return [astra.prepare_fused_add_rmsnorm(xs[i], r, ws[i], 1e-5) for i in range(n)], [r, xs, ws], {1}
    compare(build, 16 if dtype == torch.float32 else 1, passes=1)


@pytest.mark.gpu
@pytest.mark.parametrize("T,D,n", [(1, 8, 2), (16, 4096, 4), (3, 1000, 5), (256, 14336, 9), (300, 14336, 3), (40, 264, 66), (7, 1001, 4)])
@pytest.mark.parametrize("shared", ["out", "input", "nothing", "output is read next"])
def test_activations(T, D, n, shared):
    def build():
        mk = maker(T + D, torch.bfloat16)
        if shared == "output is read next":  # a call's output is the first half of the next one's input
            bufs = [mk(2 * T, 2 * D) for _ in range(2)]
            return [astra.prepare_silu_and_mul(bufs[1 - i % 2].view(4 * T, D)[:2 * T], bufs[i % 2]) for i in range(n)], bufs, {}
        inputs = [mk(T, 2 * D) for _ in range(1 if shared == "input" else n)]
        outs = [mk(T, D) for _ in range(1 if shared == "out" else n)]
        return [astra.prepare_silu_and_mul(outs[i % len(outs)], inputs[i % len(inputs)]) for i in range(n)], outs + inputs, {}
    compare(build)


@pytest.mark.gpu
@pytest.mark.parametrize("T,heads,D,n", [(1, 1, 8, 2), (16, 32, 128, 5), (3, 5, 72, 9), (64, 64, 128, 65), (256, 64, 128, 4), (20, 3, 100, 4)])
@pytest.mark.parametrize("shared", ["out", "nothing", "in place", "cascade", "no score"])
def test_merges(T, heads, D, n, shared):
    def build():
        mk = maker(T + D, torch.bfloat16)
        v = [[mk(T, heads, D), mk(T, heads, D), mk(T, heads, D)] for _ in range(n)]
        s = [[mk(T, heads, dt=torch.float32) * 10 for _ in range(3)] for _ in range(n)]
        s[0][0][0, 0] = float("-inf")
        s[1][0][0, 0] = s[1][1][0, 0] = float("-inf")
        calls = []
        for i in range(n):
            (va, vb, vo), (sa, sb, so) = v[i], s[i]
            if shared == "out":
                vo, so = v[0][2], s[0][2]
            elif shared == "in place":
                vo = va if i % 2 else vb
            elif shared == "cascade" and i > 0:  # the state so far is merged with the next one
                va, sa = v[i - 1][2], s[i - 1][2]
            calls.append(astra.prepare_merge_attn_states_lse(vo, None if shared == "no score" else so, va, sa, vb, sb))
        return calls, [t for ts in v for t in ts] + [t for ts in s for t in ts], {}
    compare(build)


@pytest.mark.gpu
@pytest.mark.parametrize("pattern", ["hidden state again", "weight is a hidden state", "same call", "two residuals", "unaligned in between"])
def test_norms_that_share_more_than_the_residual(pattern):
    T, H, n = 16, 2048, 12

    def build():
        mk = maker(5, torch.bfloat16)
        xs, r, r2, w, odd = mk(n, T, H), mk(T, H), mk(T, H), mk(H), mk(T * H + 8)
        calls = []
        for i in range(n):
            x, res, weight = xs[i], r, w
            if pattern == "hidden state again":
                x = xs[i % 3]
            elif pattern == "weight is a hidden state" and i % 4 == 3:
                weight = xs[i - 1][0]
            elif pattern == "two residuals":
                res = (r, r2)[i % 2]
            elif pattern == "unaligned in between" and i == 5:
                x = odd[8:].view(T, H)
            elif pattern == "same call":
                x = xs[0]
            calls.append(astra.prepare_fused_add_rmsnorm(x, res, weight, 1e-5))
        # a call that reads another's result carries a neighbouring value on, so its own outputs need not be equal
        return calls, [r, r2, w, xs, odd], {3, 4} if pattern in ("two residuals", "unaligned in between") else {}
    _, tensors, near = build()
    if near:
        compare(build, 1, passes=1)
        return
    # where rounding is carried on, the results are compared in value
    calls, got, _ = build()
    start = [t.clone() for t in got]
    graph = astra.CapturedCalls(calls)
    for t, s in zip(got, start):
        t.copy_(s)
    ref, want, _ = build()
    graph.replay()
    for call in ref:
        call()
    for p, q in zip(got, want):
        # each pass over a result rounds it once more: 12 roundings of 2^-8, against values of about 10
        assert (p.double() - q.double()).norm() <= 12 * 2.0 ** -8 * q.double().norm()
        assert (p != q).float().mean() < 0.01
