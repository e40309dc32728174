"""Which captured calls may run at the same time: the grouping against a brute-force conflict test (CPU),
and replays of mixed dependent and independent calls against the same calls issued in order (GPU)."""
import random
import time

import pytest
import torch

import paper_2509_07506_b200 as astra
from paper_2509_07506_b200 import binding, graphs

A = 1 << 20


def conflict(p, q):
    return any((wp or wq) and a < b + m and b < a + n for a, n, wp in p if n for b, m, wq in q if m)


@pytest.mark.parametrize("seed", range(40))
def test_calls_that_conflict_share_a_group(seed):
    rng = random.Random(seed)
    span = rng.choice((60, 400, 3000))
    calls = [tuple((rng.randrange(span), rng.choice((0, 1, 4, 9, 30)), rng.random() < 0.4) for _ in range(rng.randint(1, 5)))
             for _ in range(rng.randint(1, 25))]
    got = graphs.independent_groups(calls)
    # the finest grouping: connected components of the conflict relation
    want = list(range(len(calls)))
    for i in range(len(calls)):
        for j in range(i):
            if conflict(calls[i], calls[j]):
                a, b = want[i], want[j]
                want = [b if g == a else g for g in want]
    number = {}
    assert got == [number.setdefault(g, len(number)) for g in want]


def test_footprints_cover_every_operand():
    binding.load_library()
    fast, A = binding._fast, 1 << 20
    fp = lambda *a: list(fast.footprint(fast.prepare(*a)))  # noqa: E731
    assert fp(fast.KIND_RMSNORM, (A, 2 * A, 3 * A), (4, 64), 1e-6, 0, ()) == [(A, 512, 1), (2 * A, 512, 1), (3 * A, 128, 0)]
    assert fp(fast.KIND_SILU, (A, 2 * A), (4, 64), 0.0, 2, ()) == [(A, 1024, 1), (2 * A, 2048, 0)]
    assert fp(fast.KIND_MERGE, (A, None, 3 * A, 4 * A, 5 * A, 6 * A), (4, 8, 64), 0.0, 1, ()) == [
        (A, 4096, 1), (0, 0, 1), (3 * A, 4096, 0), (4 * A, 128, 0), (5 * A, 4096, 0), (6 * A, 128, 0)]
    assert fp(fast.KIND_ALLREDUCE_RMSNORM, (A, 2 * A, 3 * A), (4, 64), 1e-6, 0, (4 * A, 5 * A)) == [
        (A, 512, 1), (2 * A, 512, 1), (3 * A, 128, 0), (4 * A, 512, 0), (5 * A, 512, 0)]


@pytest.mark.gpu
@pytest.mark.parametrize("T", [1, 16, 200])
def test_replays_equal_the_calls_in_order(T):
    """Two chains of norms over two residuals, activations that read the first chain's result and write a
    shared buffer, merges of their own and one that reads an activation's output: three replays against the
    same calls issued one after the other, all operands bit for bit."""
    H, L = 1024, 6
    def build():
        torch.manual_seed(T)
        mk = lambda *s: torch.randn(s, device="cuda").bfloat16()  # noqa: E731
        xs, r, w = [mk(T, H) for _ in range(L)], [mk(T, H), mk(T, H)], mk(H)
        act, act2 = mk(T, H // 2), mk(T, H // 2)
        v = [mk(T, 4, 128) for _ in range(4)]
        s = [torch.randn(T, 4, device="cuda") for _ in range(3)]
        calls = []
        for i in range(L):
            calls += [astra.prepare_fused_add_rmsnorm(xs[i], r[i % 2], w, 1e-5),
                      astra.prepare_silu_and_mul(act if i % 3 else act2, xs[i if i % 2 else 0]),
                      astra.prepare_merge_attn_states_lse(v[2], s[2], v[0], s[0], v[1], s[1])]
        calls.append(astra.prepare_merge_attn_states_lse(v[3], None, act.view(T, 4, 128), s[0], v[1], s[1]))
        return calls, xs + r + [w, act, act2] + v + s
    calls_a, mem_a = build()
    calls_b, mem_b = build()
    assert max(graphs._branches(calls_a)) > 0
    graph = astra.CapturedCalls(calls_a)
    for call in calls_b:
        call()
    for _ in range(3):
        graph.replay()
        for call in calls_b:
            call()
        torch.cuda.synchronize()
        for p, q in zip(mem_a, mem_b):
            assert torch.equal(p.view(torch.int16), q.view(torch.int16))


def fake_calls(ranges):
    """Prepared norms whose x, residual and weight lie at the given addresses (nothing is launched)."""
    binding.load_library()
    ready = [binding._fast.prepare(binding._fast.KIND_RMSNORM, r, (4, 64), 1e-6, 0, ()) for r in ranges]
    return [binding.PreparedCall("norm", None, None, torch.device("cuda", 0), (), r) for r in ready]


def test_grouping_is_not_quadratic():
    """Calls that share nothing with one another: ten times as many take about ten times as long (counting the calls
    of each group one group at a time took a hundred times)."""
    def took(n):
        calls = fake_calls([(A * (3 * i + 1), A * (3 * i + 2), A * (3 * i + 3)) for i in range(n)])
        best = 1e9
        for _ in range(3):
            start = time.perf_counter()
            graphs._branches(calls)
            best = min(best, time.perf_counter() - start)
        return best
    assert took(20000) < 40 * took(2000)
