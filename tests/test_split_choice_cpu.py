"""Which circuits take two scaled fp16 parts on the tensor cores: those whose gates have entries of
one magnitude each. Steps are paired and merged with fp16 parts only, which shows the choice in the
device image."""
import copy
import math

import pytest

import circuitgen as cg
import paper_1805_01450_gb300 as q
from test_step_pairs_cpu import pairs_of
from test_step_reduces_cpu import reduces_of

PLAN = dict(n_slices=10, inner_slices=4, engine="stepwise", tensor_cores=True, order_restarts=2)


def with_gate(entries):
    """A 35-qubit circuit with a middle square-root gate replaced."""
    c = copy.deepcopy(cg.grid_circuit(5, 7, 40, 20))
    roots = [i for i, g in enumerate(c.gates) if g.kind in (cg.SQRT_X, cg.SQRT_Y)]
    i = roots[len(roots) // 2]
    c.gates[i] = cg.Gate(cg.U1, c.gates[i].q0, u=tuple(float(v) for v in entries), cycle=c.gates[i].cycle)
    return c


def merged_steps(circ, **kw):
    image = q.Plan(circ, **PLAN, **kw).image()
    return len(pairs_of(image)) + len(reduces_of(image))


def unequal(s):
    c = math.sqrt(1.0 - s * s)
    return (c, 0, -s, 0, s, 0, c, 0)


@pytest.mark.parametrize("entries,fp16", [
    (unequal(math.sqrt(0.5)), True),
    ((0.25, 0.25, 0.25, -0.25, 0.25, -0.25, 0.25, 0.25), True),       # one magnitude, scaled
    ((0, 0, 1, 0, 1, 0, 0, 0), True),                                 # zeros
    (unequal(0.6), False),
    (unequal(1 / 16), False),                                         # a ratio of 16 in one gate
    (unequal(0.06), False),
    ((1, 0, 1e-17, 0, 1e-17, 0, 1, 0), False),                        # small, but not zero
    ((2.5, 0, 2.5, 0, 2.5, 0, -2.5, 0), False),
    ((math.nan, 0, 1, 0, 1, 0, 1, 0), False),
])
def test_unequal_entries_keep_three_parts(entries, fp16):
    assert (merged_steps(with_gate(entries)) > 0) == fp16


def test_angles_that_may_change_keep_three_parts():
    # a rotation by pi / 2 has entries of one magnitude, until a gradient call gives another angle
    c = with_gate(unequal(0.6))
    i = next(i for i, g in enumerate(c.gates) if g.kind == cg.U1)
    c.gates[i] = cg.Gate(cg.RXY, c.gates[i].q0, theta=math.pi / 2, phi=0.0, param=0, cycle=c.gates[i].cycle)
    assert merged_steps(c) > 0
    assert merged_steps(c, gradient=True, mem_budget_bytes=64 << 30) == 0
