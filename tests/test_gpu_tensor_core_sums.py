"""How exact the sums of the tensor-core contractions are: circuits whose sums need no rounding
come out exact, and others within the truncation of the accumulators (the tensor cores truncate
at every multiply-add, half a unit of 2^-23 in the mean)."""
import json
import os

import numpy as np
import pytest

import circuitgen as cg
from oracle import ve as VE

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")
from test_step_pairs_cpu import pairs_of  # noqa: E402
from _program_exec import Program  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def without_t(circ):
    circ.gates = [g for g in circ.gates if g.kind != cg.T]
    return circ


@pytest.mark.parametrize("seed", (5001, 5002, 5003))
def test_sums_without_rounding_are_exact(seed):
    # H, CZ and square roots of X and Y alone: every entry is a small Gaussian integer times a
    # power of two (64 H gates: 2^-32), so a slice term has a few significant bits, not 24
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    with open(os.path.join(root, "paper_1805_01450_gb300", "orderings", f"grid8x8d40-s{seed}.json")) as f:
        d = json.load(f)
    c = without_t(cg.grid_circuit(8, 8, 40, seed))
    p = q.Plan(c, order=d["order"], slices=d["slices"], inner_slices=d["variant"]["inner_slices"], engine="stepwise",
               tensor_cores=True, mem_budget_bytes=8 << 30)
    assert len(pairs_of(p.image())) >= 1
    t = p.slice_terms(cg.random_bitstrings(64, 2, seed + 7)).cpu().numpy()
    parts = np.concatenate([t.real.ravel(), t.imag.ravel()])
    mantissa, _ = np.frexp(parts[parts != 0])
    assert mantissa.size > 0
    assert np.array_equal(mantissa * 256, np.round(mantissa * 256))


def truncations(chunks):
    """Truncations of a sum in the mean, each weighed with the part of the sum that is in by then."""
    if chunks <= 4:                        # one group: two large products a chunk
        return chunks + 0.5
    return 2.5 if chunks == 8 else 8.5     # runs of one group of two, of two groups of two


# sums of 16 to 256 entries on the streaming and the B-stationary form, alone and with a leaf
@pytest.mark.parametrize("seed,inner,longest", [(11, 5, 8), (12, 5, 7), (13, 5, 6), (2, 5, 7)])
def test_long_sums_vs_oracle(seed, inner, longest):
    c = cg.grid_circuit(6, 7, 40, seed)
    p = q.Plan(c, n_slices=10, inner_slices=inner, engine="stepwise", tensor_cores=True, plan_trials=16,
               mem_budget_bytes=32 << 30)
    image = p.image()
    pairs = pairs_of(image)
    forms = [pr["g"] for pr in pairs]
    taken = {int(pr[f]) for pr in pairs for f in ("producer", "consumer")}
    forms += [g for i, g in enumerate(Program(image).gemms) if int(g["nk"]) > 0 and i not in taken]
    assert max(int(g["nk"]) for g in forms) >= longest
    bound = sum(truncations(max(1, (1 << int(g["nk"])) // 16)) for g in forms) * 2.0 ** -24
    x = cg.random_bitstrings(42, 1, seed + 7)[0]
    terms = p.slice_terms([x]).cpu().numpy()[0].astype(np.complex128)
    ids = np.argsort(-np.abs(terms))[:8]
    ref = VE.slice_terms(c, x, p.order, p.slices, slice_ids=ids)
    err = np.linalg.norm(terms[ids] - ref) / np.linalg.norm(ref)
    # every step's truncation in one direction, and 2^-20 for the roundings of the program's FP32 sums
    assert err < bound + 2.0 ** -20


# gates whose small entry is a sixteenth or less of the large one: seven of them put entries of a
# tensor 2^-28 below its largest. The error counts against the terms themselves
@pytest.mark.parametrize("small", (1 / 16, 1 / 30, 1 / 200))
@pytest.mark.parametrize("r,c_,d,seed,k,inner", [(6, 6, 40, 7066, 8, 2), (5, 7, 40, 25, 10, 4)])
def test_unequal_gates_relative_to_the_terms(r, c_, d, seed, k, inner, small):
    c = cg.grid_circuit(r, c_, d, seed)
    roots = [i for i, g in enumerate(c.gates) if g.kind in (cg.SQRT_X, cg.SQRT_Y)]
    large = (1.0 - small * small) ** 0.5
    for i in roots[len(roots) // 4::max(1, len(roots) // 12)][:7]:
        c.gates[i] = cg.Gate(cg.U1, c.gates[i].q0, u=(large, 0.0, -small, 0.0, small, 0.0, large, 0.0), cycle=c.gates[i].cycle)
    base = q.Plan(cg.grid_circuit(r, c_, d, seed), n_slices=k, inner_slices=inner, engine="stepwise", tensor_cores=True,
                  order_restarts=2)
    p = q.Plan(c, order=base.order, slices=base.slices, inner_slices=inner, engine="stepwise", tensor_cores=True)
    assert p.info["n_gemm_steps"] >= 1 and p.step_traffic(0)[1] == 3
    x = cg.random_bitstrings(r * c_, 1, seed + 1)[0]
    terms = p.slice_terms([x]).cpu().numpy()[0].astype(np.complex128)
    ids = np.argsort(-np.abs(terms))[:6]
    ref = VE.slice_terms(c, x, p.order, p.slices, slice_ids=ids)
    assert np.linalg.norm(terms[ids] - ref) < 1e-5 * np.linalg.norm(ref)
