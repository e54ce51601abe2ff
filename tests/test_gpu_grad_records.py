"""The shared-memory gradient kernel's records, loaded two phases ahead: programs of very few phases,
phases of more records than threads, staged and unstaged launches, against the state-vector adjoint."""
import numpy as np
import pytest

import circuitgen as cg
from oracle import statevector as SV

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")


@pytest.mark.parametrize("r,c_,d,k,nb", [(2, 1, 1, 0, 3), (2, 2, 2, 0, 3), (2, 2, 4, 2, 4), (3, 4, 12, 0, 2),
                                         (4, 4, 14, 2, 200)])
def test_records_two_phases_ahead(r, c_, d, k, nb):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = cg.rotation_circuit(r, c_, d, 51)
    n = r * c_
    p = q.Plan(c, gradient=True, n_slices=k)
    xs = cg.random_bitstrings(n, nb, 52)
    a, g = (t.cpu().numpy() for t in p.amplitude_grad(xs))
    tol = 1e-5 * 2.0 ** (-n / 2)
    for i in (0, nb - 1):
        a_ref, g_ref = SV.sv_adjoint_grad(c, xs[i])
        assert abs(a[i] - a_ref) < tol
        assert np.max(np.abs(g[i] - g_ref)) < tol
