"""Work items stacked in a CTA of the fused engine: every warp count per item, passes that are full,
short and single, parts of the slice range and open outputs, against calls of one bitstring (sums
are exact, so the bits are the same) and the oracle."""
import numpy as np
import pytest

import circuitgen as cg
from oracle import ve as VE

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")


@pytest.mark.parametrize("warps", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("r,c_,d,seed,k,inner,nb", [
    (3, 3, 8, 1003, 0, 0, 400),        # a few items per SM
    (4, 4, 10, 1001, 4, 1, 1000),      # passes of full groups
    (5, 6, 20, 4001, 8, 1, 23),
    (6, 6, 25, 2001, 12, 5, 5),        # shared memory bounds the groups
])
def test_stacked_items(r, c_, d, seed, k, inner, nb, warps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cg.grid_circuit(r, c_, d, seed)
    n = r * c_
    p = q.Plan(c, n_slices=k, inner_slices=inner, engine="fused", warps_per_item=warps)
    xs = cg.random_bitstrings(n, nb, seed + 1)
    amps = p.amplitude(xs).cpu().numpy()
    for i in (0, nb // 2, nb - 1):
        assert np.array_equal(amps[i:i + 1], p.amplitude(xs[i:i + 1]).cpu().numpy())
    terms = p.slice_terms(xs).cpu().numpy()
    first, count = (1 << k) // 3, (1 << k) // 2 + 1
    count = min(count, (1 << k) - first)
    assert np.array_equal(p.slice_terms(xs, slice_begin=first, slice_count=count).cpu().numpy(), terms[:, first:first + count])
    tol = 1e-5 * 2.0 ** (-n / 2)
    ids = np.random.default_rng(seed).choice(1 << k, min(4, 1 << k), replace=False)
    ref = VE.slice_terms(c, xs[nb - 1], p.order, p.slices, slice_ids=ids)
    assert np.max(np.abs(terms[nb - 1, ids] - ref)) < tol


def test_stacked_items_open_outputs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cg.grid_circuit(4, 4, 10, 1001)
    p = q.Plan(c, n_slices=2, engine="fused", warps_per_item=4, open_qubits=[0, 5, 15])
    xs = cg.random_bitstrings(16, 800, 7)
    amps = p.amplitude(xs).cpu().numpy()
    for i in (0, 799):
        assert np.array_equal(amps[i:i + 1], p.amplitude(xs[i:i + 1]).cpu().numpy())
