"""Bytes that launches move: those of their contractions, without the tensor that two contractions
in one launch keep on the chip."""
import ctypes

import pytest

import circuitgen as cg
import paper_1805_01450_gb300 as q
from _program_exec import Program
from test_step_pairs_cpu import pairs_of, ranks
from test_step_reduces_cpu import reduces_of, small_plan

UNARY = 1


@pytest.mark.parametrize("args", [(6, 7, 32, 27, 6, 3), (5, 7, 40, 20, 10, 4), (6, 7, 40, 3, 8, 2)])
def test_merged_steps_leave_out_the_inner_tensor(args):
    p = small_plan(*args)
    image = p.image()
    steps = Program(image).steps

    def own(i):
        ra, rb = ranks(steps[i])
        return 8 * ((1 << ra) + (0 if int(steps[i]["flags"]) & UNARY else 1 << rb) + (1 << int(steps[i]["rc"])))

    merged = {int(r["producer"]): (int(r["producer"]), int(r["consumer"])) for r in pairs_of(image)}
    merged.update({int(r["consumer"]): (int(r["producer"]), int(r["consumer"])) for r in reduces_of(image)})
    assert merged
    gone = {s for pair in merged.values() for s in pair} - set(merged)
    for i in range(len(steps)):
        if i in gone:
            continue
        got, parts = p.step_traffic(i)
        assert parts == 2
        if i in merged:
            first, second = merged[i]
            assert got == own(first) + own(second) - 16 * (1 << int(steps[first]["rc"]))
        else:
            assert got == own(i)


def test_errors():
    p = q.Plan(cg.grid_circuit(3, 3, 4, 1))
    b = ctypes.c_double()
    assert q.lib().qvx_step_traffic(None, 0, ctypes.byref(b), None) == q.QVX_EINVAL
    assert q.lib().qvx_step_traffic(p._h, -1, ctypes.byref(b), None) == q.QVX_EINVAL
    assert q.lib().qvx_step_traffic(p._h, 1 << 20, ctypes.byref(b), None) == q.QVX_EINVAL
    assert q.lib().qvx_step_traffic(p._h, 0, None, None) == q.QVX_EINVAL
    assert p.step_traffic(0)[1] == 0
