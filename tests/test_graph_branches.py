"""Which captured calls may run at the same time: the grouping against a brute-force conflict test (CPU),
and replays of mixed dependent and independent calls against the same calls issued in order (GPU)."""
import ctypes
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


def test_memory_with_two_addresses_keeps_the_calls_in_order(monkeypatch):
    """Only where the driver says of every range that it is the plain allocators' does an address stand for memory;
    anything else (mapped by hand, imported, host memory) may be mapped twice, and the calls stay in one branch."""
    allocations = {}  # start -> (size, plain)
    asked = []

    @ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_uint, ctypes.POINTER(ctypes.c_int), ctypes.POINTER(ctypes.c_void_p), ctypes.c_uint64)
    def query(n, which, out, address):
        assert [which[i] for i in range(n)] == [10, 11, 12]
        asked.append(address)
        for start, (size, plain) in allocations.items():
            if start <= address < start + size:
                for i, v in enumerate((plain, start, size)):
                    ctypes.cast(out[i], ctypes.POINTER(ctypes.c_uint64))[0] = v
                return 0
        return 1
    monkeypatch.setattr(graphs, "_pointer_attributes", lambda: ctypes.cast(query, ctypes.c_void_p).value)
    calls = fake_calls([(A + 4096 * i, 2 * A + 4096 * i, 3 * A) for i in range(20)])
    allocations.update({A: (A, 1), 2 * A: (A, 1), 3 * A: (A, 1)})
    assert max(graphs._branches(calls)) == 1 and len(asked) == 3
    allocations[2 * A] = (A, 0)                       # mapped by hand
    assert graphs._branches(calls) == [0] * 20
    allocations[2 * A] = (4096 * 19 + 100, 1)         # the last range ends beyond the allocation
    assert graphs._branches(calls) == [0] * 20
    del allocations[3 * A]                            # the driver does not know the address
    assert graphs._branches(calls) == [0] * 20
    monkeypatch.setattr(graphs, "_pointer_attributes", lambda: None)
    assert graphs._branches(calls) == [0] * 20


class At:
    """A [rows, width] float32 array at an address."""

    def __init__(self, address, shape):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f4", "data": (address, False), "version": 3, "strides": None}


@pytest.mark.gpu
def test_memory_mapped_twice_is_not_captured_into_two_branches():
    driver = pytest.importorskip("cuda.bindings.driver")

    def ok(result):
        assert int(result[0]) == 0, result
        return result[1] if len(result) == 2 else result[1:]
    torch.zeros(1, device="cuda")
    where = driver.CUmemLocation()
    where.type, where.id = driver.CUmemLocationType.CU_MEM_LOCATION_TYPE_DEVICE, 0
    prop = driver.CUmemAllocationProp()
    prop.type, prop.location = driver.CUmemAllocationType.CU_MEM_ALLOCATION_TYPE_PINNED, where
    size = ok(driver.cuMemGetAllocationGranularity(prop, driver.CUmemAllocationGranularity_flags.CU_MEM_ALLOC_GRANULARITY_MINIMUM))
    access = driver.CUmemAccessDesc()
    access.location, access.flags = where, driver.CUmemAccess_flags.CU_MEM_ACCESS_FLAGS_PROT_READWRITE
    handle = ok(driver.cuMemCreate(size, prop, 0))
    mapped = []
    for _ in range(2):
        at = ok(driver.cuMemAddressReserve(size, 0, 0, 0))
        ok(driver.cuMemMap(at, size, 0, handle, 0))
        ok(driver.cuMemSetAccess(at, size, [access], 1))
        mapped.append(int(at))
    T, H = 64, 256
    one, two = (torch.as_tensor(At(p, (T, H)), device="cuda") for p in mapped)
    r, w, out = torch.zeros(T, H, device="cuda"), torch.ones(H, device="cuda"), torch.empty(T, H // 2, device="cuda")
    calls = [astra.prepare_fused_add_rmsnorm(one, r, w, 1e-5), astra.prepare_silu_and_mul(out, two)]
    assert graphs.independent_groups([c.footprint() for c in calls]) == [0, 1]   # by their addresses
    assert graphs._branches(calls) == [0, 0]
    graph = astra.CapturedCalls(calls)
    one.copy_(torch.randn(T, H, device="cuda"))
    r.zero_()
    graph.replay()
    torch.cuda.synchronize()
    want = torch.empty_like(out)
    astra.astra_silu_and_mul(want, one)
    assert torch.equal(out, want)
    del graph
    torch.cuda.synchronize()
    for p in mapped:
        ok(driver.cuMemUnmap(p, size))
        ok(driver.cuMemAddressFree(p, size))
    ok(driver.cuMemRelease(handle))


def test_one_branch_on_request(monkeypatch):
    calls = fake_calls([(A * (3 * i + 1), A * (3 * i + 2), A * (3 * i + 3)) for i in range(6)])
    monkeypatch.setattr(graphs, "_pointer_attributes", lambda: None)
    monkeypatch.setattr(binding._fast, "one_address_each", lambda calls, query: True)
    assert sorted(graphs._branches(calls)) == [0, 0, 0, 1, 1, 1]
    assert graphs._branches(calls, 1) == [0] * 6
    assert sorted(graphs._branches(calls, 3)) == [0, 0, 1, 1, 2, 2]
