"""The arena of plans with merged steps: every operand and result of a launch lies within it, and
the results that no launch stores take no room in it."""
import json
import os

import pytest

import circuitgen as cg
import paper_1805_01450_gb300 as q
from _program_exec import A_LEAF, B_LEAF, Program
from test_step_pairs_cpu import pairs_of, ranks
from test_step_reduces_cpu import reduces_of, small_plan

UNARY = 1


def recorded(seed, tensor_cores=True):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    with open(os.path.join(root, "paper_1805_01450_gb300", "orderings", f"grid8x8d40-s{seed}.json")) as f:
        d = json.load(f)
    return q.Plan(cg.grid_circuit(8, 8, 40, seed), order=d["order"], slices=d["slices"],
                  inner_slices=d["variant"]["inner_slices"], engine="stepwise", tensor_cores=tensor_cores,
                  mem_budget_bytes=64 << 30)


def launched_extent(p):
    """The largest entry that a launch reads or writes."""
    image = p.image()
    prog = Program(image)
    steps = prog.steps
    unstored = {int(r["producer"]) for r in list(pairs_of(image)) + reduces_of(image)}
    end = 0
    for s, st in enumerate(steps):
        if s not in unstored:   # a pair writes its consumer's result, a merged step its own
            end = max(end, int(st["c_off"]) + (1 << int(st["rc"])))
        ra, rb = ranks(st)
        for leaf, off, rank in ((A_LEAF, "a_off", ra), (B_LEAF, "b_off", rb)):
            flags = int(st["flags"])
            if flags & leaf or (off == "b_off" and flags & UNARY):
                continue
            producer = max((i for i in range(s) if int(steps[i]["c_off"]) == int(st[off]) and int(steps[i]["rc"]) == rank), default=None)
            if producer is not None and producer in unstored:
                continue
            end = max(end, int(st[off]) + (1 << rank))
    return end, int(prog.h["arena_elems"])


PLANS = [(6, 7, 32, 27, 6, 3), (5, 7, 40, 20, 10, 4), (7, 7, 30, 17, 6, 3), (6, 6, 36, 32, 6, 3), (6, 7, 40, 3, 8, 2)]


@pytest.mark.parametrize("args", PLANS)
def test_launches_stay_within_the_arena(args):
    p = small_plan(*args)
    end, whole = launched_extent(p)
    assert 0 < end <= p.info["arena_bytes"] // 8 <= whole


@pytest.mark.parametrize("seed", (5001, 5002, 5003))
def test_unstored_results_take_no_room(seed):
    p, plain = recorded(seed), recorded(seed, tensor_cores=False)
    end, whole = launched_extent(p)
    assert end <= p.info["arena_bytes"] // 8 < whole
    # the largest results of these programs are never stored: less than 0.6 of the plain arena
    assert p.info["arena_bytes"] < 0.6 * plain.info["arena_bytes"]
    assert p.workspace_bytes(1) < plain.workspace_bytes(1)
