"""GPU parity of steps merged into the consumer of their result, and of pairs of steps, against
the oracle, over the summed-column counts, batch and column splits that the small plans have."""
import numpy as np
import pytest

import circuitgen as cg
from oracle import ve as VE

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")
from test_step_reduces_cpu import PLANS, reduces_of, small_plan  # noqa: E402


@pytest.mark.parametrize("args", PLANS)
@pytest.mark.parametrize("budget", [1 << 30, 24 << 20])   # all work items at once, one or two at a time
def test_merged_steps_vs_oracle(args, budget):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r, c_, d, seed, k, inner = args
    base = small_plan(*args)
    c = cg.grid_circuit(r, c_, d, seed)
    p = q.Plan(c, order=base.order, slices=base.slices, inner_slices=inner, engine="stepwise", tensor_cores=True,
               mem_budget_bytes=budget)
    assert reduces_of(p.image())
    n = r * c_
    xs = cg.random_bitstrings(n, 2, seed + 1)
    terms = p.slice_terms(xs).cpu().numpy()
    ids = np.random.default_rng(seed).choice(1 << k, 5, replace=False)
    for i, x in enumerate(xs):
        ref = VE.slice_terms(c, x, p.order, p.slices, slice_ids=ids)
        assert np.max(np.abs(terms[i, ids] - ref)) < 1e-5 * 2.0 ** (-n / 2)
