"""Which captured calls share a launch: the library's decision for every way of sharing operands, on both sides of each limit
(no GPU: addresses are only compared), and the order of capture where addresses do not tell memory apart."""
import ctypes

import pytest
import torch

from paper_2509_07506_b200 import binding, graphs

A = 1 << 30  # tensors are A apart, so that none of them meet unless they are meant to
BF16, FP16, FP32 = 0, 1, 2


def plan(kind, calls, ext, dtype=BF16):
    """Calls per launch; calls: the pointer arguments of each in the order of its entry point."""
    lib, fast = binding.load_library(), binding._fast
    flat = [p for c in calls for p in (*c, *(0,) * (6 - len(c)))]
    counts, launches = (ctypes.c_int32 * max(1, len(calls)))(), ctypes.c_int32(-1)
    st = lib.astra_plan_run(getattr(fast, "KIND_" + kind), ctypes.c_int32(len(calls)), (ctypes.c_void_p * max(1, len(flat)))(*flat),
                            (ctypes.c_int64 * 4)(*ext, *(0,) * (4 - len(ext))), ctypes.c_int(dtype), counts, ctypes.byref(launches))
    assert st == 0
    got = list(counts[:launches.value])
    assert sum(got) == len(calls)
    return got


def silus(n, **fixed):
    return [(fixed.get("out", (2 * i + 1) * A), fixed.get("inp", (2 * i + 2) * A)) for i in range(n)]


def norms(n, r=A, w=2 * A):
    return [((i + 3) * A, r, w) for i in range(n)]


def merges(n, score=A // 2):
    return [tuple(x for k in (1, 2, 3) for x in ((3 * i + k) * A, (3 * i + k) * A + score)) for i in range(n)]  # (vo, so, va, sa, vb, sb)


@pytest.mark.parametrize("n,want", [(0, []), (1, [1]), (2, [2]), (3, [3]), (64, [64]), (65, [64, 1]), (130, [64, 64, 2])])
def test_calls_of_one_launch(n, want):
    assert plan("SILU", silus(n), (16, 4096)) == want
    assert plan("RMSNORM", norms(n), (16, 4096)) == want
    assert plan("MERGE", merges(n), (16, 32, 128)) == want


def test_shared_operands_of_activations():
    ext = (16, 4096)
    out_bytes = 16 * 4096 * 2
    assert plan("SILU", silus(5, inp=99 * A), ext) == [5]
    assert plan("SILU", silus(5, out=99 * A), ext) == [5]                          # the same output: in order within a thread
    chained = [((i + 2) * A, (i + 1) * A) for i in range(4)]                       # each reads the previous one's output
    assert plan("SILU", chained, ext) == [1] * 4
    c = silus(4)
    assert plan("SILU", [c[0], (c[0][0] + out_bytes, c[1][1]), *c[2:]], ext) == [4]         # outputs side by side
    assert plan("SILU", [c[0], (c[0][0] + out_bytes - 32, c[1][1]), *c[2:]], ext) == [1, 3]  # outputs that meet in part
    assert plan("SILU", [c[0], c[1], (c[0][1], c[2][1]), c[3]], ext) == [2, 2]              # writes what an earlier one reads
    assert plan("SILU", [c[0], (c[1][0], c[1][0]), *c[2:]], ext) == [1, 1, 2]               # refused by the entry point
    assert plan("SILU", [c[0], (c[1][0] + 8, c[1][1]), *c[2:]], ext) == [1, 1, 2]           # 8-byte aligned: no form of a run
    assert plan("SILU", [c[0], (c[1][0] + 16, c[1][1]), *c[2:]], ext) == [4]


def test_shared_operands_of_norms():
    ext, x = (16, 4096), lambda i: (i + 3) * A  # noqa: E731
    c = norms(6)
    assert plan("RMSNORM", [(x(i), A, 2 * A if i % 2 else 90 * A) for i in range(6)], ext) == [6]   # weights shared or not
    assert plan("RMSNORM", [(x(i), (1 if i % 2 else 80) * A, 2 * A) for i in range(6)], ext) == [1] * 6  # two residuals in turn
    assert plan("RMSNORM", [*c[:3], *c[:3]], ext) == [3, 3]                                         # a hidden state again
    assert plan("RMSNORM", [c[0], c[1], (x(2), A, x(1)), *c[3:]], ext) == [2, 4]                    # the weight is a hidden state
    assert plan("RMSNORM", [c[0], c[1], (x(2), A, A + 64), *c[3:]], ext) == [2, 1, 3]               # ... or the residual: refused
    assert plan("RMSNORM", [c[0], (x(1) + 16, A, 2 * A), *c[2:]], ext) == [1, 1, 4]                 # accesses of another width
    assert plan("RMSNORM", [c[0], (x(1) + 8, A, 2 * A), *c[2:]], ext) == [1, 1, 4]


def test_shared_operands_of_merges():
    ext, c = (16, 32, 128), merges(4)
    assert plan("MERGE", [(c[0][0], c[0][1], *m[2:]) for m in c], ext) == [4]                # one output
    assert plan("MERGE", [(m[2], *m[1:]) for m in c], ext) == [4]                            # in place
    assert plan("MERGE", [(m[0], 0, *m[2:]) for m in c], ext) == [4]                         # no score
    cascade = [c[0], *((m[0], m[1], p[0], p[1], *m[4:]) for p, m in zip(c, c[1:]))]
    assert plan("MERGE", cascade, ext) == [1] * 4
    assert plan("MERGE", [c[0], (*c[1][:3], c[0][1], *c[1][4:]), *c[2:]], ext) == [1, 3]     # reads only a score of the first
    assert plan("MERGE", [c[0], (*c[1][:3], c[1][3] + 2, *c[1][4:]), *c[2:]], ext) == [1, 1, 2]  # a score at 2 bytes: refused
    shifted = (c[1][2] + 32, *c[1][1:])                                                      # in place, but for 32 bytes: refused
    assert plan("MERGE", [c[0], shifted, *c[2:]], ext) == [1, 1, 2]


@pytest.mark.parametrize("kind,few,many", [("SILU", 1 << 21, 1 << 22), ("RMSNORM", 1 << 22, None), ("MERGE", 1 << 20, 1 << 21)])
@pytest.mark.parametrize("dtype", [BF16, FP16, FP32])
def test_sizes(kind, few, many, dtype):
    calls = {"SILU": silus, "RMSNORM": norms, "MERGE": merges}[kind]
    width = (2048,) if kind != "MERGE" else (16, 128)
    per_row = 2048 * (2 if dtype == FP32 else 1)
    for limit, n in ((few, 2), (few, 3), (many, 4), (many, 9)):
        if limit is None:  # norms gain at every size
            assert plan(kind, calls(n), (1 << 14, *width), dtype) == [n]
            continue
        rows = limit // per_row
        assert plan(kind, calls(n), (rows, *width), dtype) == [n]
        assert plan(kind, calls(n), (rows + 1, *width), dtype) == [1] * n
    assert plan(kind, calls(4), (0, *width), dtype) == [1] * 4


@pytest.mark.parametrize("T,H,dtype,want", [(16, 8, BF16, 4), (16, 4, BF16, 1), (37, 8192, BF16, 4), (75, 8192, BF16, 4), (75, 4096, FP32, 4),
                                            (16, 8200, BF16, 1), (16, 8208, BF16, 1), (75, 8208, BF16, 1), (75, 4104, FP32, 1),
                                            (16, 11008, BF16, 1), (75, 4100, BF16, 1), (75, 4104, BF16, 1), (75, 4096, BF16, 4)])
def test_widths_of_norms(T, H, dtype, want):
    assert plan("RMSNORM", norms(4), (T, H), dtype) == ([4] if want == 4 else [1] * 4)


def test_memory_with_two_addresses_is_captured_call_by_call(monkeypatch):
    binding.load_library()
    fast = binding._fast
    calls = [binding.PreparedCall("call", None, None, torch.device("cuda", 0), (),
                                  fast.prepare(fast.KIND_SILU, (A * (2 * i + 1), A * (2 * i + 2)), (4, 64), 0.0, 0, ())) for i in range(6)]
    monkeypatch.setattr(graphs, "_pointer_attributes", lambda: None)
    monkeypatch.setattr(fast, "one_address_each", lambda calls, query: False)
    assert graphs._plan(calls, 2) == [(0, [c]) for c in calls]
    monkeypatch.setattr(fast, "one_address_each", lambda calls, query: True)
    assert sorted(b for b, _ in graphs._plan(calls, 2)) == [0, 0, 0, 1, 1, 1]
