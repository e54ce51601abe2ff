"""Register-tiled steps of the stepwise engine: several blocks of tiles per CTA, items of fewer tiles
than a CTA has threads, swapped operands and 8 x 4 tiles, against calls of one bitstring (the same
bits, whatever the blocks per CTA) and the persistent engine's kernels."""
import numpy as np
import pytest

import circuitgen as cg
from _program_exec import Program

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")

CASES = [
    # rows, cols, depth, seed, sliced, open, bitstrings
    (4, 4, 10, 1001, 0, 0, 9),
    (6, 6, 25, 2001, 3, 1, 70),
    (7, 7, 30, 3001, 2, 2, 128),      # 8 blocks of tiles per CTA
    (6, 7, 36, 5, 6, 4, 2),
]


@pytest.mark.parametrize("r,c_,d,seed,k,inner,nb", CASES)
def test_blocks_of_tiles(r, c_, d, seed, k, inner, nb):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cg.grid_circuit(r, c_, d, seed)
    n = r * c_
    kw = dict(n_slices=k, inner_slices=inner, mem_budget_bytes=16 << 30)
    s = q.Plan(c, engine="stepwise", tensor_cores=False, plan_trials=8, **kw)
    tiles = [t for t in Program(s.image()).rtsteps if t["rm"] + t["rn"] > 0]
    if d == 30:
        square = [t for t in tiles if t["rm"] == 2 and t["rn"] == 2 and t["nt"] >= 8]
        assert any(t["a_cb"] > t["b_cb"] for t in square) and any(t["a_cb"] < t["b_cb"] for t in square)
        assert any(t["rm"] + t["rn"] == 5 for t in tiles) and any(t["nt"] < 8 for t in tiles)
    xs = cg.random_bitstrings(n, nb, seed + 1)
    a = s.slice_terms(xs).cpu().numpy()
    for i in (0, nb // 2, nb - 1):
        assert np.array_equal(a[i:i + 1], s.slice_terms(xs[i:i + 1]).cpu().numpy())
    p = q.Plan(c, order=s.order, slices=s.slices, inner_slices=inner, engine="persistent", mem_budget_bytes=1 << 30)
    tol = 1e-5 * 2.0 ** (-n / 2)
    assert np.max(np.abs(a[:2] - p.slice_terms(xs[:2]).cpu().numpy())) < tol
