"""The persistent engine's register tiles (every tile shape of the plans, tile indexes within the
first and second table and above both, work items in several passes, slice ranges) against the
stepwise engine's kernels and, where it is quick, the oracle."""
import numpy as np
import pytest

import circuitgen as cg
from _program_exec import Program
from oracle import ve as VE

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")

CASES = [
    # rows, cols, depth, seed, sliced, open, budget, bitstrings
    (4, 4, 10, 1001, 2, 0, 1 << 30, 5),
    (6, 6, 25, 2001, 6, 2, 1 << 30, 2),
    (6, 6, 25, 2001, 6, 0, 2 << 20, 3),       # a few work items at a time
    (7, 7, 30, 3001, 6, 2, 256 << 20, 1),
    (6, 7, 36, 5, 6, 4, 1 << 30, 1),          # tile indexes of more than 16 bits
]


@pytest.mark.parametrize("r,c_,d,seed,k,inner,budget,nb", CASES)
def test_persistent_tiles(r, c_, d, seed, k, inner, budget, nb):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cg.grid_circuit(r, c_, d, seed)
    n = r * c_
    kw = dict(n_slices=k, inner_slices=inner, mem_budget_bytes=budget)
    p = q.Plan(c, engine="persistent", **kw)
    s = q.Plan(c, order=p.order, slices=p.slices, inner_slices=inner, engine="stepwise", mem_budget_bytes=budget)
    tiles = [t for t in Program(p.image()).rtsteps if t["rm"] + t["rn"] > 0]
    assert all(t["rm"] <= 2 and t["rn"] <= 2 for t in tiles)
    if d == 36:
        assert max(int(t["nt"]) for t in tiles) > 16
    if d == 30:
        assert 8 < max(int(t["nt"]) for t in tiles)
    xs = cg.random_bitstrings(n, nb, seed + 1)
    tol = 1e-5 * 2.0 ** (-n / 2)
    a = p.slice_terms(xs).cpu().numpy()
    assert np.max(np.abs(a - s.slice_terms(xs).cpu().numpy())) < tol
    first, count = (1 << k) // 3, (1 << k) // 2 + 1
    part = p.slice_terms(xs, slice_begin=first, slice_count=count).cpu().numpy()
    assert np.array_equal(part, a[:, first:first + count])
    if n <= 36:
        ids = np.random.default_rng(seed).choice(1 << k, min(4, 1 << k), replace=False)
        ref = VE.slice_terms(c, xs[0], p.order, p.slices, slice_ids=ids)
        assert np.max(np.abs(a[0, ids] - ref)) < tol
