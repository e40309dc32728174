"""Workloads for timing the library through its public entry points.

Each case is one pass of what a serving program asks of this library: a decode step's small calls, a
prefill step's large ones, the all-reduce forms of tensor-parallel ranks, strided operands, ragged
widths, every storage type, and the three ways of issuing a call (directly, prepared, or replayed from a
CUDA graph).  Shapes come from ``paper_2509_07506_b200.workloads``, the test suite and ``bench.py``.

``listed()`` gives the named cases, ``draw(rng)`` another one of the same ranges; ``prepare`` builds the
tensors a caller has in hand, ``run`` issues the calls, ``exact`` gives their results in 64 bits, ``work``
states the unavoidable bytes and operations, ``tolerance`` how far another correct implementation may
be off.
"""
from __future__ import annotations

import math

import torch

import paper_2509_07506_b200 as astra
from paper_2509_07506_b200 import workloads as wl

_TORCH = {"bf16": torch.bfloat16, "fp16": torch.float16, "fp32": torch.float32}
_ELEM = {"bf16": 2, "fp16": 2, "fp32": 4}
EPS = 1e-5
DEVICE = "cuda"

# hidden and intermediate widths, heads and head sizes that the repository's configurations name
HIDDEN = (2048, 4096, 5120, 8192, 11008, 14336, 16384)
INTERMEDIATE = (4096, 5120, 8192, 11008, 12288, 14336)
HEADS = (8, 32, 40, 64)
HEAD_DIMS = (64, 80, 128, 256)
MAX_BYTES = 1.17e9          # about the largest listed case


def listed():
    return [
        # one decode step's norm, called directly: latency of a call on very little data
        {"name": "norm_decode", "op": "rmsnorm", "T": 16, "H": 4096, "dtype": "bf16", "form": "plain"},
        # the activation of a batched decode step
        {"name": "silu_decode_batch", "op": "silu", "T": 128, "D": 14336, "dtype": "bf16", "form": "plain"},
        # merge of prefix and suffix attention for a few hundred tokens, some of them without a prefix
        {"name": "merge_chunk", "op": "merge", "T": 512, "heads": 32, "D": 128, "dtype": "bf16", "empty": 0.01,
         "form": "plain"},
        # a chunked-prefill norm of a wide model in half precision
        {"name": "norm_chunk_wide", "op": "rmsnorm", "T": 1024, "H": 8192, "dtype": "fp16", "form": "plain"},
        # a long prefill over a width that is not a multiple of eight
        {"name": "norm_prefill_ragged", "op": "rmsnorm", "T": 16384, "H": 4100, "dtype": "bf16", "form": "plain"},
        # the three operations of a long prefill one after the other (what bench.py times)
        {"name": "chain_prefill", "op": "chain", "T": 8192, "H": 4096, "D": 14336, "heads": 32, "head_dim": 128,
         "dtype": "bf16", "form": "plain"},
        # all layers of a decode step replayed from a CUDA graph
        {"name": "graph_decode", "op": "graph", "T": 16, "H": 4096, "D": 14336, "heads": 32, "head_dim": 128,
         "layers": 32, "dtype": "bf16", "form": "graph"},
        # the all-reduce folded into a decode step's norm, eight ranks
        {"name": "allreduce_decode", "op": "allreduce", "T": 16, "H": 4096, "parts": 8, "dests": 1, "dtype": "bf16",
         "form": "plain"},
        # a rank's row block of a prefill, results stored to every rank's buffers (two-shot form)
        {"name": "two_shot_prefill", "op": "allreduce", "T": 2048, "H": 8192, "parts": 4, "dests": 4, "dtype": "bf16",
         "form": "plain"},
        # merge with the head-major scores that attention kernels return, values as they come
        {"name": "merge_head_major", "op": "merge", "T": 2048, "heads": 40, "D": 128, "dtype": "fp16", "empty": 0.01,
         "form": "strided"},
        # merge of split attention results kept in single precision
        {"name": "merge_fp32", "op": "merge", "T": 4096, "heads": 32, "D": 128, "dtype": "fp32", "empty": 0.0,
         "form": "plain"},
        # an activation whose odd width leaves every row at another alignment
        {"name": "silu_odd_width", "op": "silu", "T": 1000, "D": 14337, "dtype": "fp16", "form": "plain"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, common):
    """Mostly a width that models have; one time in four any width of that range."""
    return rng.choice(common) if rng.random() < 0.75 else rng.randint(min(common), max(common))


def draw(rng):
    while True:
        case = {"op": rng.choice(("rmsnorm", "rmsnorm", "silu", "silu", "merge", "merge", "allreduce", "chain", "graph")),
                "T": _log_int(rng, 1, 16384), "dtype": rng.choice(("bf16", "bf16", "bf16", "fp16", "fp16", "fp32"))}
        form = rng.choice(("plain", "plain", "strided"))
        if case["op"] == "rmsnorm":
            case.update(H=_width(rng, HIDDEN), form=form)
        elif case["op"] == "silu":
            case.update(D=_width(rng, INTERMEDIATE), form=form)
        elif case["op"] == "merge":
            case.update(heads=rng.choice(HEADS), D=rng.choice(HEAD_DIMS), empty=rng.choice((0.0, 0.01, 0.05)), form=form)
        elif case["op"] == "allreduce":
            parts = rng.choice((2, 4, 8))
            case.update(H=_width(rng, HIDDEN), parts=parts, dests=rng.choice((1, 1, parts)), form="plain")
        elif case["op"] == "chain":
            case.update(H=rng.choice(HIDDEN), D=rng.choice(INTERMEDIATE), heads=rng.choice(HEADS), head_dim=128,
                        form=rng.choice(("plain", "prepared")))
        else:
            case.update(T=_log_int(rng, 1, 256), H=rng.choice((2048, 4096, 5120, 8192)), D=rng.choice(INTERMEDIATE),
                        heads=rng.choice(HEADS), head_dim=128, layers=rng.randint(4, 32), form="graph")
            if case["dtype"] == "fp32":
                case["dtype"] = "bf16"
        if work(case)["bytes"] <= MAX_BYTES:
            return case


# ---- inputs ---------------------------------------------------------------------------------------

def _randn(g, shape, dtype, mean=0.0, std=1.0):
    t = torch.randn(shape, generator=g, device=DEVICE, dtype=torch.float32)
    return t.mul_(std).add_(mean).to(_TORCH[dtype])


def _rows(t, pad):
    """The same rows as a slice of a wider buffer (pitch = width + pad)."""
    wide = torch.empty((*t.shape[:-1], t.shape[-1] + pad), dtype=t.dtype, device=t.device)
    view = wide[..., :t.shape[-1]]
    view.copy_(t)
    return view


def _scores(g, T, heads, empty):
    s = torch.rand((T, heads), generator=g, device=DEVICE) * 30.0 - 10.0
    if empty > 0.0:
        s.masked_fill_(torch.rand((T, heads), generator=g, device=DEVICE) < empty, float("-inf"))
    return s


def _norm_tensors(g, T, H, dtype):
    return _randn(g, (T, H), dtype), _randn(g, (T, H), dtype), _randn(g, (H,), dtype, 1.0, 0.1)


def _silu_tensors(g, T, D, dtype):
    return _randn(g, (T, 2 * D), dtype, 0.0, 2.0), torch.empty((T, D), dtype=_TORCH[dtype], device=DEVICE)


def _merge_tensors(g, T, heads, D, dtype, empty):
    va, vb = _randn(g, (T, heads, D), dtype), _randn(g, (T, heads, D), dtype)
    sa, sb = _scores(g, T, heads, empty), _scores(g, T, heads, empty)
    return va, sa, vb, sb, torch.empty_like(va), torch.empty_like(sa)


def prepare(case, seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    op, T, dtype, form = case["op"], case["T"], case["dtype"], case["form"]
    st = {"op": op, "form": form}
    if op == "rmsnorm":
        x, r, w = _norm_tensors(g, T, case["H"], dtype)
        if form == "strided":  # slices of a projection's output; results into buffers of their own
            x, r = _rows(x, 128), _rows(r, 128)
            st.update(y=torch.empty((T, case["H"]), dtype=x.dtype, device=DEVICE),
                      ro=torch.empty((T, case["H"]), dtype=x.dtype, device=DEVICE))
        st.update(x=x, r=r, w=w)
    elif op == "silu":
        inp, out = _silu_tensors(g, T, case["D"], dtype)
        if form == "strided":  # gate and up as two tensors
            st.update(gate=inp[:, :case["D"]].contiguous(), up=inp[:, case["D"]:].contiguous())
        st.update(inp=inp, out=out)
    elif op == "merge":
        va, sa, vb, sb, vo, so = _merge_tensors(g, T, case["heads"], case["D"], dtype, case["empty"])
        if form == "strided":  # scores stored [heads, T], as attention kernels return them
            sa, sb, so = (t.t().contiguous().t() for t in (sa, sb, so))
        st.update(va=va, sa=sa, vb=vb, sb=sb, vo=vo, so=so)
    elif op == "allreduce":
        n, d = case["parts"], case["dests"]
        parts = [_randn(g, (T, case["H"]), dtype, 0.0, n ** -0.5) for _ in range(n)]
        _, r, w = _norm_tensors(g, T, case["H"], dtype)
        ys = [torch.empty_like(r) for _ in range(d)]
        st.update(parts=parts, r=r, w=w, ys=ys, rs=[r] + [torch.empty_like(r) for _ in range(d - 1)])
    elif op == "chain":
        x, r, w = _norm_tensors(g, T, case["H"], dtype)
        inp, out = _silu_tensors(g, T, case["D"], dtype)
        va, sa, vb, sb, vo, so = _merge_tensors(g, T, case["heads"], case["head_dim"], dtype, 0.0)
        st.update(x=x, r=r, w=w, inp=inp, out=out, va=va, sa=sa, vb=vb, sb=sb, vo=vo, so=so)
        if form == "prepared":
            st["calls"] = [astra.prepare_fused_add_rmsnorm(x, r, w, EPS), astra.prepare_silu_and_mul(out, inp),
                           astra.prepare_merge_attn_states_lse(vo, so, va, sa, vb, sb)]
    else:  # graph: per layer norm, merge, norm, activation; one residual stream, activation buffers reused by all layers
        L = case["layers"]
        xs = torch.empty((2 * L, T, case["H"]), dtype=_TORCH[dtype], device=DEVICE)
        r = torch.empty((T, case["H"]), dtype=_TORCH[dtype], device=DEVICE)
        ws = _randn(g, (2 * L, case["H"]), dtype, 1.0, 0.1)
        inp, out = _silu_tensors(g, T, case["D"], dtype)
        va, sa, vb, sb, vo, so = _merge_tensors(g, T, case["heads"], case["head_dim"], dtype, 0.0)
        xs.zero_()
        r.zero_()
        calls = []
        for i in range(L):
            calls += [astra.prepare_fused_add_rmsnorm(xs[2 * i], r, ws[2 * i], EPS),
                      astra.prepare_merge_attn_states_lse(vo, so, va, sa, vb, sb),
                      astra.prepare_fused_add_rmsnorm(xs[2 * i + 1], r, ws[2 * i + 1], EPS),
                      astra.prepare_silu_and_mul(out, inp)]
        st["graph"] = astra.CapturedCalls(calls)
        # capturing runs the calls once, so the inputs are filled afterwards
        xs.copy_(torch.randn(xs.shape, generator=g, device=DEVICE))
        r.copy_(torch.randn(r.shape, generator=g, device=DEVICE))
        st.update(xs=xs, ws=ws, r=r, inp=inp, out=out, va=va, sa=sa, vb=vb, sb=sb, vo=vo, so=so)
    return st


# ---- one pass -------------------------------------------------------------------------------------

def _issue(st):
    op, form = st["op"], st["form"]
    if form == "prepared":
        for call in st["calls"]:
            call()
    elif op == "rmsnorm":
        if form == "strided":
            astra.astra_fused_add_rmsnorm_ex(st["y"], st["ro"], st["x"], st["r"], st["w"], EPS)
        else:
            astra.astra_fused_add_rmsnorm(st["x"], st["r"], st["w"], EPS)
    elif op == "silu":
        if form == "strided":
            astra.astra_silu_and_mul_ex(st["out"], st["gate"], st["up"])
        else:
            astra.astra_silu_and_mul(st["out"], st["inp"])
    elif op == "merge":
        if form == "strided":
            astra.astra_merge_attn_states_lse_ex(st["vo"], st["so"], st["va"], st["sa"], st["vb"], st["sb"])
        else:
            astra.astra_merge_attn_states_lse(st["vo"], st["so"], st["va"], st["sa"], st["vb"], st["sb"])
    elif op == "allreduce":
        if len(st["ys"]) > 1:
            astra.astra_fused_allreduce_add_rmsnorm_ex(st["ys"], st["rs"], st["r"], st["parts"], st["w"], EPS)
        else:
            astra.astra_fused_allreduce_add_rmsnorm(st["ys"][0], st["r"], st["parts"], st["w"], EPS)
    elif op == "chain":
        astra.astra_fused_add_rmsnorm(st["x"], st["r"], st["w"], EPS)
        astra.astra_silu_and_mul(st["out"], st["inp"])
        astra.astra_merge_attn_states_lse(st["vo"], st["so"], st["va"], st["sa"], st["vb"], st["sb"])
    else:
        st["graph"].replay()


def run(st):
    _issue(st)
    op = st["op"]
    if op == "rmsnorm":
        return [st["y"], st["ro"]] if st["form"] == "strided" else [st["x"], st["r"]]
    if op == "silu":
        return [st["out"]]
    if op == "merge":
        return [st["vo"], st["so"]]
    if op == "allreduce":
        return [st["ys"], st["rs"]]
    if op == "chain":
        return [st["x"], st["r"], st["out"], st["vo"], st["so"]]
    return [st["xs"], st["r"], st["out"], st["vo"], st["so"]]


# ---- the same pass in 64 bits -----------------------------------------------------------------------

def _exact_norm(x, r, w):
    """(normalised rows, unrounded residual) of the add and RMSNorm; all arithmetic in 64 bits."""
    s = x.double() + r.double()
    return s * torch.rsqrt((s * s).mean(dim=1, keepdim=True) + EPS) * w.double(), s


def _exact_silu(inp):
    a, b = inp.double().chunk(2, dim=1)
    return a * torch.sigmoid(a) * b


def _exact_merge(va, sa, vb, sb):
    sa, sb = sa.double(), sb.double()
    m = torch.maximum(sa, sb)
    m = m.masked_fill(m == float("-inf"), 0.0)
    ea, eb = torch.exp(sa - m), torch.exp(sb - m)
    total = ea + eb
    share = torch.where(total > 0, 1.0 / total, total)   # two empty states merge to an empty one
    v = (ea * share).unsqueeze(2) * va.double() + (eb * share).unsqueeze(2) * vb.double()
    return v, m + torch.log(total)


def exact(case, seed):
    """What ``run`` returns for these inputs, in 64 bits.  The residual stream of the graph case is kept in
    its storage type between the layers, as the caller's buffer keeps it."""
    st = prepare(case, seed)
    op = case["op"]
    if op == "rmsnorm":
        return list(_exact_norm(st["x"], st["r"], st["w"]))
    if op == "silu":
        return [_exact_silu(st["inp"])]
    if op == "merge":
        return list(_exact_merge(st["va"], st["sa"], st["vb"], st["sb"]))
    if op == "allreduce":
        total = st["parts"][0].double()
        for p in st["parts"][1:]:
            total = total + p.double()
        y, r = _exact_norm(total, st["r"], st["w"])
        return [[y] * len(st["ys"]), [r] * len(st["rs"])]
    silu, (vo, so) = _exact_silu(st["inp"]), _exact_merge(st["va"], st["sa"], st["vb"], st["sb"])
    if op == "chain":
        return [*_exact_norm(st["x"], st["r"], st["w"]), silu, vo, so]
    ys, r = [], st["r"]
    for x, w in zip(st["xs"], st["ws"]):
        y, s = _exact_norm(x, r, w)
        ys.append(y)
        r = s.to(st["r"].dtype)
    return [torch.stack(ys), s, silu, vo, so]


# ---- what a pass cannot do without ------------------------------------------------------------------

def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: per norm element one add for the
    residual (and for each further partial), two for the square sum and two for the scaling; five per
    SiLU element (exponential, add, reciprocal, two multiplies); three per merged element."""
    op, T, e = case["op"], case["T"], _ELEM[case["dtype"]]
    if op == "rmsnorm":
        return {"bytes": wl.rmsnorm_bytes(T, case["H"], e), "flops": 5 * T * case["H"]}
    if op == "silu":
        return {"bytes": wl.silu_bytes(T, case["D"], e), "flops": 5 * T * case["D"]}
    if op == "merge":
        return {"bytes": wl.merge_bytes(T, case["heads"], case["D"], e), "flops": 3 * T * case["heads"] * case["D"]}
    if op == "allreduce":
        n, d = case["parts"], case["dests"]
        return {"bytes": wl.two_shot_rmsnorm_bytes(T, case["H"], n, d, d, e), "flops": (4 + n) * T * case["H"]}
    norm = (wl.rmsnorm_bytes(T, case["H"], e), 5 * T * case["H"])
    silu = (wl.silu_bytes(T, case["D"], e), 5 * T * case["D"])
    merge = (wl.merge_bytes(T, case["heads"], case["head_dim"], e), 3 * T * case["heads"] * case["head_dim"])
    if op == "chain":
        return {"bytes": norm[0] + silu[0] + merge[0], "flops": norm[1] + silu[1] + merge[1]}
    L = case["layers"]
    return {"bytes": L * (2 * norm[0] + silu[0] + merge[0]), "flops": L * (2 * norm[1] + silu[1] + merge[1])}


def tolerance(case):
    """Arithmetic is binary32 with one rounding to the storage type at each store, so an output is off
    its 64-bit value by that rounding: a 2-norm of 1.7e-3 for bf16 and 2.1e-4 for fp16; 0.5e-7 to 1e-7
    for fp32, where the approximate exponential, reciprocal and square root show instead (largest single
    differences 3.9e-3, 4.9e-4 and 2.7e-7).  Four times those, and a little for the second rounding of
    results that a further pass updates in place."""
    return {"bf16": {"rel": 6.8e-3, "max": 1.6e-2}, "fp16": {"rel": 8.4e-4, "max": 2e-3},
            "fp32": {"rel": 4e-7, "max": 2e-6}}[case["dtype"]]
