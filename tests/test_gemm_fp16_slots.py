"""The prefill GEMM's fp16 weight tiles, their barriers modelled on the CPU.

A group of dequantiser warps takes every GROUPS-th stage; its stages use its
OPS / GROUPS weight slots in turn.  For a stage of fp16 weights every warp waits
until the slot is free, one of them asks for the copy, every warp waits for the
copy on a parity of its barrier and then arrives for the MMAs, which free the
slot.  The model walks every order in which warps, copies and MMAs can move and
looks for a state in which a warp waits for ever.  The numbers of warps, slots
and barriers are those of the kernel's source.
"""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2607_14618_gb300", "csrc", "polyq_gemm.cu")


def _configs():
    """(name, warps of a group, weight slots of a group, w16 barriers of a group)."""
    text = open(SRC).read()
    dim = re.search(r"uint64_t bar_w16\[C::(\w+)\]", text).group(1)
    out = []
    for name, args in re.findall(r"using (Cfg\d+) = Cfg<([^>]*)>;", text):
        _, _, _, ops, _, _, groups, _ = (int(a) for a in args.split(","))
        out.append((name, 12 // groups, ops // groups, {"OPS": ops, "GROUPS": groups}[dim] // groups))
    return out


def _passes(done, parity):
    """mbarrier.try_wait.parity on a barrier with `done` phases complete."""
    return (done & 1) != parity


def _stuck_state(warps, slots, bars, stages):
    """A reachable state with work left that nothing can move, or None.

    State: per warp its stage and step (0: wait for the slot, 1: wait for the
    copy, 2: finished); phases done of each w16 barrier and of each slot's
    `free` barrier; copies under way per w16 barrier; arrivals per slot.  Warp 0
    asks for the copies."""
    start = (((0, 0),) * warps, (0,) * bars, (0,) * slots, (0,) * bars, (0,) * slots)
    seen, todo = {start}, [start]
    while todo:
        state = todo.pop()
        pcs, w16, free, copies, arrived = state
        moves = []

        def put(t, i, v):
            return t[:i] + (v,) + t[i + 1:]

        for w, (j, step) in enumerate(pcs):
            if step == 2:
                continue
            s, b = j % slots, j % bars
            if step == 0 and _passes(free[s], (j // slots + 1) & 1):
                c = put(copies, b, copies[b] + 1) if w == 0 else copies
                moves.append((put(pcs, w, (j, 1)), w16, free, c, arrived))
            if step == 1 and _passes(w16[b], (j // bars) & 1):
                nxt = (j, 2) if j + 1 == stages else (j + 1, 0)
                moves.append((put(pcs, w, nxt), w16, free, copies, put(arrived, s, arrived[s] + 1)))
        for b in range(bars):
            if copies[b]:  # a copy lands
                moves.append((pcs, put(w16, b, w16[b] + 1), free, put(copies, b, copies[b] - 1), arrived))
        for s in range(slots):
            if arrived[s] == warps:  # the stage's MMAs have run
                moves.append((pcs, w16, put(free, s, free[s] + 1), copies, put(arrived, s, 0)))
        if not moves and any(step != 2 for _, step in pcs):
            return state
        for m in moves:
            if m not in seen:
                seen.add(m)
                todo.append(m)
    return None


@pytest.mark.parametrize("name,warps,slots,bars", _configs(), ids=[c[0] for c in _configs()])
def test_no_warp_waits_for_ever(name, warps, slots, bars):
    assert _stuck_state(warps, slots, bars, stages=3 * slots) is None


def test_model_finds_a_barrier_shared_by_two_slots():
    """One barrier for a group's two slots gets two phases ahead of a slow warp."""
    assert _stuck_state(warps=4, slots=2, bars=1, stages=4) is not None
    assert _stuck_state(warps=4, slots=2, bars=2, stages=6) is None
