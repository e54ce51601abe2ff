"""info["n_gemm_steps"] counts the contractions that launches run on the tensor cores."""
import pytest

import circuitgen as cg
import paper_1805_01450_gb300 as q
from _program_exec import Program
from test_step_pairs_cpu import pairs_of
from test_step_reduces_cpu import reduces_of


# the first has merged steps and not one plain contraction that qualifies
@pytest.mark.parametrize("r,c_,d,seed,k,inner,kw", [
    (6, 6, 40, 9, 10, 4, dict(plan_trials=4)), (5, 7, 40, 20, 10, 4, dict(order_restarts=2)), (6, 7, 40, 2, 10, 5, {}),
    (6, 6, 40, 7066, 8, 2, {}), (4, 4, 10, 1, 2, 0, {})])
def test_count(r, c_, d, seed, k, inner, kw):
    c = cg.grid_circuit(r, c_, d, seed)
    p = q.Plan(c, n_slices=k, inner_slices=inner, engine="stepwise", tensor_cores=True, **kw)
    image = p.image()
    pairs, reds = pairs_of(image), reduces_of(image)
    steps = {int(r[f]) for r in pairs for f in ("producer", "consumer")} | {int(r["producer"]) for r in reds}
    steps |= {i for i, g in enumerate(Program(image).gemms) if int(g["nk"]) > 0 and i not in {int(r["consumer"]) for r in reds}}
    assert p.info["n_gemm_steps"] == len(steps)
    assert (p.info["n_gemm_steps"] > 0) == (d == 40)
    simt = q.Plan(c, order=p.order, slices=p.slices, inner_slices=inner, engine="stepwise")
    assert simt.info["n_gemm_steps"] == 0
