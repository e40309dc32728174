"""The extension's own checks of direct calls: what is not the ordinary case is left to the binding's
Python route (nothing launched, None returned), so that every refusal keeps its error."""
import os
import subprocess
import sys
import threading
import time
import timeit

import pytest
import torch

from paper_2509_07506_b200 import binding


@pytest.fixture(scope="module")
def fast():
    binding.load_library()
    return binding._fast


def test_operands_that_are_not_cuda_tensors_are_left_to_the_binding(fast):
    t = torch.zeros((2, 8), dtype=torch.bfloat16)
    for bad in (t, None, 3, object()):
        assert fast.rmsnorm(bad, t, t[0], 1e-6, None) is None
        assert fast.silu(t, bad, None) is None
        assert fast.merge(t, None, bad, t, t, t, None) is None
        assert fast.allreduce_rmsnorm(bad, t, [t], t[0], 1e-6, None) is None
        assert fast.rmsnorm_ex(t, t, bad, t, t[0], 1e-6, None) is None
        assert fast.silu_ex(t, bad, t, None) is None
        assert fast.merge_ex(t, t, bad, t, t, t, None) is None
        assert fast.allreduce_rmsnorm_ex([t], [t], bad, [t], t[0], 1e-6, None) is None
    with pytest.raises(TypeError):
        fast.rmsnorm(t, t)


@pytest.mark.parametrize("missing", [False, True])
def test_another_torch_does_without_direct_calls(monkeypatch, fast, missing):
    """An extension of another torch release, or none, is left out with a warning; the library, prepared calls and
    the binding's own route need neither."""
    t = torch.zeros((2, 8), dtype=torch.bfloat16)
    try:
        with monkeypatch.context() as m:
            m.setattr(binding, "_lib", None)
            if missing:
                m.setattr(binding, "TORCHCALL_PATH", binding.TORCHCALL_PATH + ".none")
            else:
                m.setattr(torch, "__version__", "0.1.2")
            with pytest.warns(RuntimeWarning, match="missing" if missing else "built for torch"):
                binding.load_library()
            assert binding._fast.silu(t, t, None) is None and binding._fast.build_id()
            assert type(binding._fast.silu) is not type(binding._fast.build_id)
            with pytest.raises(TypeError, match="CUDA"):
                binding.astra_fused_add_rmsnorm(t, t, t[0], 1e-6)
    finally:
        binding._lib = None
        binding.load_library()
    assert type(binding._fast.silu) is type(binding._fast.build_id)


def test_leaving_a_call_to_the_binding_costs_no_more_than_the_call(fast):
    """A refusal comes on top of the Python route on every such call; as a C++ exception it cost 20 to 40 empty
    calls of the extension."""
    t = torch.zeros((2, 8), dtype=torch.bfloat16)
    best = lambda f: min(timeit.repeat(f, number=1000, repeat=20))  # noqa: E731
    assert best(lambda: fast.rmsnorm(t, t, t, 1e-6, None)) < 8 * best(lambda: fast.build_id())


class Undirect:
    """The extension with every direct call left to the binding."""

    def __init__(self, fast):
        self.fast = fast

    def __getattr__(self, name):
        if name.split("_ex")[0] in ("rmsnorm", "silu", "merge", "allreduce_rmsnorm"):
            return lambda *a: None
        return getattr(self.fast, name)


class Sub(torch.Tensor):
    pass


def outcome(call, *args):
    try:
        call(*args)
        torch.cuda.synchronize()
        return None
    except Exception as e:  # noqa: BLE001 - the type and text are what is compared
        return type(e), str(e)


def norm(T=3, H=64, dtype=torch.bfloat16):
    mk = lambda *s: torch.randn(s, device="cuda").to(dtype)  # noqa: E731
    return mk(T, H), mk(T, H), mk(H)


def calls():
    """(name of the function, arguments) of ordinary, unusual and refused calls, drawn anew each time."""
    b = binding
    x, r, w = norm()
    inp, out = torch.randn(3, 64, device="cuda").half(), torch.zeros(3, 32, device="cuda", dtype=torch.float16)
    va, vb, vo = (torch.randn(3, 4, 16, device="cuda") for _ in range(3))
    sa, sb, so = (torch.randn(3, 4, device="cuda") for _ in range(3))
    wide = torch.randn(3, 96, device="cuda").bfloat16()
    side = torch.cuda.Stream()
    many = [x.clone() for _ in range(17)]
    ys = [torch.zeros_like(x) for _ in range(2)]
    yield from [
        (b.astra_fused_add_rmsnorm, (x, r, w, 1e-6)), (b.astra_fused_add_rmsnorm, (x, r, w, 1)),
        (b.astra_fused_add_rmsnorm, (x, r, torch.nn.Parameter(w, requires_grad=False), 1e-6, side)),
        (b.astra_fused_add_rmsnorm, (x.as_subclass(Sub), r, w, 1e-6)),
        (b.astra_fused_add_rmsnorm, (x, r, w, torch.tensor(1e-6))), (b.astra_fused_add_rmsnorm, (x, r, w, "no")),
        (b.astra_fused_add_rmsnorm, (x, x, w, 1e-6)), (b.astra_fused_add_rmsnorm, (x, r.float(), w, 1e-6)),
        (b.astra_fused_add_rmsnorm, (x.t(), r, w, 1e-6)), (b.astra_fused_add_rmsnorm, (x, r[:2], w, 1e-6)),
        (b.astra_fused_add_rmsnorm, (x, r.cpu(), w, 1e-6)), (b.astra_fused_add_rmsnorm, (x, r, w[:8], 1e-6)),
        (b.astra_fused_add_rmsnorm, (x[0], r[0], w, 1e-6)), (b.astra_fused_add_rmsnorm, (x.double(), r, w, 1e-6)),
        (b.astra_fused_add_rmsnorm, (x[:0], r[:0], w, 1e-6)), (b.astra_fused_add_rmsnorm, (x, r, w, 1e-6, "stream")),
        (b.astra_silu_and_mul, (out, inp)), (b.astra_silu_and_mul, (inp[:, :32], inp)), (b.astra_silu_and_mul, (out, inp[:, 1:])),
        (b.astra_silu_and_mul, (out.bfloat16(), inp)), (b.astra_silu_and_mul, (inp.view(-1)[:96].view(3, 32), inp)),
        (b.astra_merge_attn_states_lse, (vo, so, va, sa, vb, sb)), (b.astra_merge_attn_states_lse, (vo, None, va, sa, vb, sb)),
        (b.astra_merge_attn_states_lse, (vo, sa, va, sa, vb, sb)), (b.astra_merge_attn_states_lse, (vo, so.half(), va, sa, vb, sb)),
        (b.astra_merge_attn_states_lse, (vo, so, va, sa.t(), vb, sb)), (b.astra_merge_attn_states_lse, (vo[:2], so, va, sa, vb, sb)),
        (b.astra_fused_allreduce_add_rmsnorm, (ys[0], r, [x, x], w, 1e-6)),
        (b.astra_fused_allreduce_add_rmsnorm, (ys[0], r, iter((x, x)), w, 1e-6)),
        (b.astra_fused_allreduce_add_rmsnorm, (ys[0], r, many, w, 1e-6)), (b.astra_fused_allreduce_add_rmsnorm, (ys[0], r, [], w, 1e-6)),
        (b.astra_fused_allreduce_add_rmsnorm, (ys[0], r, (x, ys[0]), w, 1e-6)),
        (b.astra_fused_allreduce_add_rmsnorm_ex, (ys, (r, x.clone()), r, [x, x], w, 1e-6)),
        (b.astra_fused_allreduce_add_rmsnorm_ex, (ys, [r], r, [x, x.half()], w, 1e-6)),
        (b.astra_fused_allreduce_add_rmsnorm_ex, (ys + ys, [r], r, [x], w, 1e-6)),
        (b.astra_fused_add_rmsnorm_ex, (ys[0], ys[1], wide[:, :64], wide[:, 32:], w, 1e-6)),
        (b.astra_fused_add_rmsnorm_ex, (wide[:, :64], r, wide[:, :64], r, w, 1e-6)),
        (b.astra_fused_add_rmsnorm_ex, (ys[0], ys[1], wide[:, ::2][:, :32], r, w, 1e-6)),
        (b.astra_fused_add_rmsnorm_ex, (ys[0], ys[1], x[:1].expand(3, 64), r, w, 1e-6)),
        (b.astra_silu_and_mul_ex, (ys[0], wide[:, :64], wide[:, 32:])), (b.astra_silu_and_mul_ex, (ys[0], wide, x)),
        (b.astra_silu_and_mul_ex, (ys[0][:1], x[:1], r[:1])),
        (b.astra_merge_attn_states_lse_ex, (vo, so.t().contiguous().t(), va, sa.t().contiguous().t(), vb, sb)),
        (b.astra_merge_attn_states_lse_ex, (vo, None, va, sa[:, :1].expand(3, 4), vb, sb)),
        (b.astra_merge_attn_states_lse_ex, (vo, so[:, :1].expand(3, 4), va, sa, vb, sb)),
        (b.astra_merge_attn_states_lse_ex, (vo, so, va.transpose(1, 2), sa, vb, sb)),
    ]


@pytest.mark.gpu
def test_both_routes_accept_refuse_and_compute_alike(monkeypatch, fast):
    """Every call through the extension's checks and with them switched off: the same results in all the
    operands, or the same error."""
    def run(direct):
        seen = []
        if not direct:
            monkeypatch.setattr(binding, "_fast", Undirect(fast))
        torch.manual_seed(5)
        for fn, args in calls():
            torch.cuda.synchronize()
            err = outcome(fn, *args)
            flat = [t for a in args for t in (a if isinstance(a, (list, tuple)) else [a]) if isinstance(t, torch.Tensor)]
            seen.append((fn.__name__, err, [t.detach().as_subclass(torch.Tensor).cpu().contiguous() for t in flat]))
        return seen
    a, b = run(True), run(False)
    assert sum(err is None for _, err, _ in a) > 12 and sum(err is not None for _, err, _ in a) > 20
    for i, ((name, ea, ta), (_, eb, tb)) in enumerate(zip(a, b)):
        assert ea == eb, (i, name, ea, eb)
        for p, q in zip(ta, tb):
            assert torch.equal(p.reshape(-1).view(torch.uint8), q.reshape(-1).view(torch.uint8)), (i, name)


@pytest.mark.gpu
def test_wrappers_and_modes_take_the_bindings_own_route(fast):
    x, r, w = norm()
    assert fast.rmsnorm(x, r, w, 1e-6, None) == 0
    assert fast.rmsnorm(x.as_subclass(Sub), r, w, 1e-6, None) is None
    with torch.device("cuda"):  # a torch-function mode
        assert fast.rmsnorm(x, r, w, 1e-6, None) is None
    seen = []
    torch.func.vmap(lambda v: (seen.append(fast.rmsnorm(v, r, w, 1e-6, None)), v)[1])(torch.stack([x, x]))
    assert seen == [None]
    torch.cuda.synchronize()


@pytest.mark.gpu
def test_plain_calls_keep_the_interpreter_lock(fast):
    """Beside a thread that computes in Python, a call that gave the lock up would wait for it for a whole switch
    interval; so many calls in a row would take `n` of them."""
    x, r, w = norm()
    va, sa = torch.randn(3, 4, 16, device="cuda"), torch.randn(3, 4, device="cuda")
    vo, so, y = torch.empty_like(va), torch.empty_like(sa), torch.empty_like(x)
    inp, out = torch.randn(3, 64, device="cuda"), torch.empty(3, 32, device="cuda")

    def every():
        binding.astra_fused_add_rmsnorm(x, r, w, 1e-6)
        binding.astra_silu_and_mul(out, inp)
        binding.astra_merge_attn_states_lse(vo, so, va, sa, va, sa)
        binding.astra_fused_allreduce_add_rmsnorm(y, r, [x, x], w, 1e-6)

    every()
    torch.cuda.synchronize()
    done = threading.Event()

    def compute():
        while not done.is_set():
            pass
    interval, n = 0.05, 20
    before = sys.getswitchinterval()
    other = threading.Thread(target=compute, daemon=True)
    sys.setswitchinterval(interval)
    try:
        other.start()
        start = time.perf_counter()
        for _ in range(n // 4):
            every()
        took = time.perf_counter() - start
    finally:
        done.set()
        sys.setswitchinterval(before)
        other.join()
    torch.cuda.synchronize()
    assert took < n * interval / 4  # the lock may still be asked for once or twice in between


@pytest.mark.gpu
def test_threads_in_a_call_at_the_interpreters_end():
    """A daemon thread that is in an unlocked launch when the interpreter ends is unwound when it comes for the
    lock; the process ends with its own status all the same."""
    code = """if True:
        import sys, threading, time, torch
        import paper_2509_07506_b200 as astra
        x, r, w = (torch.zeros(s, device="cuda") for s in ((2, 64), (2, 64), 64))
        ys, rs = [torch.zeros_like(x) for _ in range(2)], [torch.zeros_like(x) for _ in range(2)]
        def work():
            while True:
                astra.astra_fused_add_rmsnorm_ex(ys[0], rs[0], x, r, w, 1e-6)
                astra.astra_fused_allreduce_add_rmsnorm_ex(ys, rs, r, [x], w, 1e-6)
        for _ in range(4):
            threading.Thread(target=work, daemon=True).start()
        time.sleep(0.5)
        torch.cuda.synchronize()
        sys.exit(7)
    """
    root = os.path.dirname(os.path.dirname(os.path.abspath(binding.__file__)))
    done = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert done.returncode == 7, (done.returncode, done.stderr[-2000:])
