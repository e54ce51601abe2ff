"""The two operand splits of the tensor-core contractions: two scaled fp16 parts for circuits
whose gate entries are alike in size, three bf16 parts for the others, each against the FP64
oracle on circuits with some gates multiplied by powers of two (which scale every slice term
exactly, so the tolerance scales with them)."""
import numpy as np
import pytest

import circuitgen as cg
from oracle import ve as VE

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")

MATRICES = {cg.SQRT_X: ((0.5, 0.5), (0.5, -0.5), (0.5, -0.5), (0.5, 0.5)),
            cg.SQRT_Y: ((0.5, 0.5), (-0.5, -0.5), (0.5, 0.5), (0.5, 0.5))}


def scaled(circ, every, exponent):
    """The circuit with every `every`-th square-root gate as a U1 gate times 2^exponent, and
    the exponent of the whole amplitude's factor."""
    out, seen, total = cg.Circuit(circ.n_qubits, [], circ.rows, circ.cols, circ.depth), 0, 0
    for g in circ.gates:
        if g.kind in MATRICES:
            seen += 1
            if seen % every == 0:
                u = tuple(float(c) * 2.0 ** exponent for e in MATRICES[g.kind] for c in e)
                out.gates.append(cg.Gate(cg.U1, g.q0, u=u, cycle=g.cycle))
                total += exponent
                continue
        out.gates.append(g)
    return out, total


# every gate entry stays within 2^-4 ... 2 (fp16 parts): unscaled, scaled down and up; one entry
# range outside (bf16 parts): far down, far up
@pytest.mark.parametrize("every,exponent", [(1 << 30, 0), (7, -2), (9, 1), (40, -14), (40, 12)])
@pytest.mark.parametrize("r,c_,d,seed,k,inner", [(6, 6, 40, 7066, 8, 2), (5, 6, 40, 19, 8, 2)])
def test_scaled_gates_vs_oracle(r, c_, d, seed, k, inner, every, exponent):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    base = cg.grid_circuit(r, c_, d, seed)
    n = r * c_
    circ, total = scaled(base, every, exponent)
    ref_plan = q.Plan(base, n_slices=k, inner_slices=inner, engine="stepwise", tensor_cores=True)
    p = q.Plan(circ, order=ref_plan.order, slices=ref_plan.slices, inner_slices=inner, engine="stepwise", tensor_cores=True)
    assert p.info["n_gemm_steps"] >= 1 and abs(total) < 120
    xs = cg.random_bitstrings(n, 2, seed + 1)
    terms = p.slice_terms(xs).cpu().numpy().astype(np.complex128)
    ids = np.random.default_rng(seed).choice(1 << k, 6, replace=False)
    for i, x in enumerate(xs):
        ref = VE.slice_terms(circ, x, p.order, p.slices, slice_ids=ids)
        assert np.max(np.abs(terms[i, ids] - ref)) < 1e-5 * 2.0 ** (-n / 2) * 2.0 ** total
