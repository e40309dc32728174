"""Replaying a fixed sequence of calls from a CUDA graph.

For decode-sized batches every call of this library is bound by launch cost, not by the GPU: a
call costs 2.0-2.5 us of host time for 1-2 us of device time.  A sequence of prepared
calls on fixed tensors (a layer's add+norm, activation and merge, say) can be captured once into a
CUDA graph and replayed with a single launch; the kernels keep their programmatic-dependent-launch
edges inside the graph, so each one's prologue (and its L2 prefetch) overlaps the previous one's tail, and
calls of one kind and shape that follow one another share a launch (``csrc/call_runs.cuh``).
torch's graph object is used for capture and replay: device plumbing, no arithmetic.
"""
from __future__ import annotations

import ctypes
from typing import List, Optional, Sequence, Tuple

import torch

from . import binding
from .binding import PreparedCall

# Calls that share no memory one of them writes are captured into parallel branches, two at most.  Each call
# of a dependent sequence is a chain of latencies (launch, first bytes, reduction, completion) that leaves
# most of the GPU idle while it waits; a second sequence fills that time.  Measured on norm, merge, norm, activation
# repeated 32 times where only the norms share a tensor (one residual), per repetition with 1 / 2 / 4 branches, the latter
# two with like calls in one launch: 4.70 / 0.71 / 0.77 us at 1 token of width 4096, 4.93 / 0.77 / 0.77 at 16, 6.40 / 1.60 /
# 1.58 at 64, 9.53 / 4.22 / 4.37 at 256, 13.2 / 9.7 / 9.7 at 512 and 26.2 / 18.0 / 20.5 at 1024 tokens.  Calls that are linked
# through their tensors, as a decoder layer's are, stay one sequence and gain nothing.
MAX_BRANCHES = 2


def independent_groups(calls: Sequence) -> List[int]:
    """A group number per call (0, 1, ... in order of first appearance) such that two calls of different
    groups touch no common byte that either of them writes.  ``calls[i]`` is the extension's struct of call i or
    the ``(address, bytes, is_written)`` ranges of it."""
    binding.load_library()
    return binding._fast.independent_groups(calls)


_driver: Optional[ctypes.CDLL] = None


def _pointer_attributes() -> Optional[int]:
    """Address of the driver's cuPointerGetAttributes, or None."""
    global _driver
    if _driver is None:
        try:
            _driver = ctypes.CDLL("libcuda.so.1")
        except OSError:
            return None
    return ctypes.cast(_driver.cuPointerGetAttributes, ctypes.c_void_p).value


def _groups(calls: Sequence[PreparedCall], most: int) -> Optional[List[int]]:
    """The group number of each call, or None where the calls are to be captured as they come: on request, where a
    call is not one of ours, or where addresses do not tell whether two calls share memory."""
    if most < 2 or len(calls) < 2 or any(type(c) is not PreparedCall for c in calls):
        return None
    ready = [c._ready for c in calls]
    return independent_groups(ready) if binding._fast.one_address_each(ready, _pointer_attributes()) else None


def _branches(calls: Sequence[PreparedCall], most: int = MAX_BRANCHES) -> List[int]:
    """The branch each call is captured into; all zeros where there is one sequence."""
    groups = _groups(calls, most)
    return [0] * len(calls) if groups is None else _branches_of(groups, most)


def _branches_of(groups: List[int], most: int) -> List[int]:
    sizes = [0] * (max(groups) + 1)
    for g in groups:
        sizes[g] += 1
    load, branch_of = [0] * min(most, len(sizes)), [0] * len(sizes)
    for g in sorted(range(len(sizes)), key=lambda g: -sizes[g]):
        branch_of[g] = min(range(len(load)), key=load.__getitem__)
        load[branch_of[g]] += sizes[g]
    return [branch_of[g] for g in groups]


def _plan(calls: Sequence[PreparedCall], most: int) -> List[Tuple[int, List[PreparedCall]]]:
    """``(branch, run)`` in the order of capture; a run is calls that are issued together.  Calls of one group keep
    their order, and those of it that follow one another and are alike form a run."""
    groups = _groups(calls, most)
    if groups is None:
        return [(0, [c]) for c in calls]
    runs, last = [], {}  # the group's latest run
    for call, group, branch in zip(calls, groups, _branches_of(groups, most)):
        run = last.get(group)
        if run is not None and run[0]._device == call._device and binding._fast.alike(run[0]._ready, call._ready):
            run.append(call)
        else:
            last[group] = run = [call]
            runs.append((branch, run))
    return runs


def _issue(run: List[PreparedCall], stream: torch.cuda.Stream) -> None:
    if len(run) == 1:
        run[0](stream)
    else:
        binding.issue_run(run, stream)


class CapturedCalls:
    """``CapturedCalls([call_a, call_b, ...])`` runs the prepared calls once eagerly on a side stream
    (so that lazy initialisation happens outside the capture), then captures them;
    ``replay()`` re-issues the whole sequence on the current stream with one launch, with the results of
    the calls issued in order: calls that depend on one another through a tensor stay in that order, and
    calls that share no written memory may run at the same time, in at most ``branches`` sequences (1: all in the
    order given, one launch each).  Calls of one kind and shape that follow one another in a sequence are issued
    together where their operands allow it; the squares of a norm's row are then summed in another order than by a
    single call, everything else is bit for bit the same.  The tensors the
    calls were prepared on are the graph's inputs and outputs.  The eager warm-up run has already
    executed every call once when the constructor returns (in-place calls such as fused_add_rmsnorm
    have then modified their operands), so fill the inputs after constructing, and refill them in
    place between replays."""

    def __init__(self, calls: Sequence[PreparedCall], device: Optional[torch.device] = None,
                 branches: int = MAX_BRANCHES):
        self.calls = list(calls)
        if not self.calls:
            raise ValueError("at least one prepared call is needed")
        self.device = device if device is not None else torch.device("cuda", torch.cuda.current_device())
        side = torch.cuda.Stream(self.device)
        side.wait_stream(torch.cuda.current_stream(self.device))
        with torch.cuda.stream(side):
            plan = _plan(self.calls, branches)
            for _, run in plan:           # warm-up outside the capture
                _issue(run, side)
            side.synchronize()
            streams = [side] + [torch.cuda.Stream(self.device) for _ in range(max(branch for branch, _ in plan))]
            self.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(self.graph, stream=side):
                for s in streams[1:]:
                    s.wait_stream(side)
                for branch, run in plan:
                    _issue(run, streams[branch])
                for s in streams[1:]:
                    side.wait_stream(s)
        torch.cuda.current_stream(self.device).wait_stream(side)

    def replay(self) -> None:
        self.graph.replay()
