"""GPU parity of every tensor-core kernel that a step may run on, against the FP64 oracle: plain
steps and steps with a leaf on their rows or columns, streaming and B-stationary, at each column
width, in one accumulator, in groups of four chunks and in several runs; and the three-part form
of the same circuits. Steps that a merged one replaces are not launched and do not count."""
import copy
import math

import numpy as np
import pytest

import circuitgen as cg
from oracle import ve as VE

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
q = pytest.importorskip("paper_1805_01450_gb300")
from _program_exec import Program  # noqa: E402
from test_step_pairs_cpu import pairs_of  # noqa: E402
from test_step_reduces_cpu import reduces_of  # noqa: E402

# most chunks of 16 summed entries whose B fits in shared memory, by real columns
RESIDENT = {2: {256: 4, 128: 8, 64: 16, 32: 32, 16: 64}, 3: {256: 2, 128: 4, 64: 8, 32: 16, 16: 32}}


def launched(image, parts):
    """(leaf side or plain, real columns, form, how the sum is accumulated) of the launches."""
    pairs, reds = pairs_of(image), reduces_of(image)
    gone = {int(r[f]) for r in list(pairs) + reds for f in ("producer", "consumer")}
    steps = [("rows" if p["leaf"]["on_rows"] else "cols", p["g"]) for p in pairs]
    steps += [("plain", g) for i, g in enumerate(Program(image).gemms) if int(g["nk"]) > 0 and i not in gone]
    out = set()
    for kind, g in steps:
        nm, nn, nk = (int(g[f]) for f in ("nm", "nn", "nk"))
        nt, chunks = 256 if nn >= 7 else 2 << nn, max(1, (1 << nk) // 16)
        bs = (1 << nm) // 128 >= 4 and chunks <= RESIDENT[parts][nt]
        how = "one" if parts == 3 or chunks <= 2 else "four" if chunks == 4 else "runs"
        out.add((kind, nt, "stationary" if bs else "streaming", how))
    return out


S, B = "streaming", "stationary"
CASES = [   # (rows, cols, depth, seed, sliced, inner), launches that the case is there for
    ((5, 7, 40, 25, 10, 4), [("cols", 256, S, "one"), ("cols", 256, S, "runs"), ("plain", 128, S, "one")]),
    ((6, 6, 36, 33, 8, 2), [("plain", 16, S, "one"), ("plain", 64, B, "one"), ("rows", 16, B, "one"), ("rows", 32, B, "one")]),
    ((5, 7, 40, 35, 10, 4), [("cols", 128, S, "runs"), ("plain", 32, B, "one"), ("rows", 128, S, "one"), ("rows", 16, S, "one")]),
    ((6, 6, 40, 16, 10, 4), [("cols", 32, B, "four"), ("plain", 256, B, "one"), ("plain", 256, B, "four"), ("plain", 256, S, "four")]),
    ((6, 6, 36, 37, 10, 4), [("cols", 32, B, "one"), ("cols", 64, S, "one"), ("plain", 64, S, "one")]),
    ((6, 6, 40, 28, 10, 4), [("cols", 64, S, "four"), ("plain", 256, S, "one"), ("rows", 32, S, "one")]),
    ((6, 6, 36, 25, 10, 4), [("cols", 128, S, "one"), ("plain", 64, S, "runs")]),
    ((6, 6, 36, 2, 8, 2), [("cols", 16, S, "one"), ("rows", 64, S, "one")]),
    ((5, 6, 40, 15, 8, 2), [("cols", 16, S, "four"), ("rows", 64, B, "one")]),
    ((5, 7, 40, 14, 8, 2), [("cols", 16, B, "one"), ("rows", 256, S, "one")]),
    ((6, 6, 40, 18, 8, 2), [("cols", 64, B, "one"), ("rows", 256, S, "runs")]),
    ((6, 6, 40, 12, 8, 2), [("cols", 256, B, "four"), ("rows", 64, S, "four")]),
    ((5, 6, 40, 9, 8, 2), [("plain", 16, B, "one")]),
    ((6, 6, 36, 15, 8, 2), [("rows", 16, S, "four")]),
    ((5, 6, 40, 8, 8, 2), [("rows", 32, S, "four")]),
    ((5, 7, 40, 18, 10, 4), [("rows", 128, B, "one")]),
    ((5, 7, 40, 5, 8, 2), [("cols", 32, S, "runs")]),
    ((5, 7, 40, 11, 10, 4), [("plain", 128, B, "one")]),
    ((5, 6, 40, 19, 10, 4), [("cols", 128, B, "one")]),
    ((5, 7, 40, 37, 8, 2), [("rows", 256, B, "one")]),
    ((6, 6, 40, 11, 10, 4), [("cols", 256, B, "one")]),
    ((5, 7, 40, 7, 10, 4), [("cols", 64, B, "four")]),
    ((5, 6, 40, 20, 8, 2), [("rows", 16, B, "four")]),
    ((6, 6, 36, 9, 8, 2), [("plain", 128, S, "runs")]),
    ((6, 6, 40, 37, 8, 2), [("cols", 64, B, "runs")]),
    ((6, 6, 40, 10, 10, 4), [("plain", 16, S, "four")]),
    ((5, 6, 40, 35, 10, 4), [("plain", 128, B, "four")]),
    ((6, 6, 40, 38, 8, 2), [("cols", 32, B, "runs")]),
    ((6, 7, 40, 8, 10, 4), [("plain", 256, S, "runs"), ("cols", 128, B, "runs")]),
    ((5, 7, 40, 5, 10, 4), [("cols", 64, S, "runs")]),
    ((5, 7, 40, 10, 8, 2), [("cols", 16, S, "runs")]),
    ((5, 7, 40, 9, 10, 4), [("rows", 32, S, "runs")]),
]
THREE_PARTS = set()   # launches of the three-part runs below


def plan(circ, args, **kw):
    return q.Plan(circ, n_slices=args[4], inner_slices=args[5], engine="stepwise", tensor_cores=True, order_restarts=2, **kw)


def unequal(circ, s):
    """The circuit with its middle square-root gate replaced by a rotation of entries c, s."""
    out = copy.deepcopy(circ)
    roots = [i for i, g in enumerate(out.gates) if g.kind in (cg.SQRT_X, cg.SQRT_Y)]
    i, c = roots[len(roots) // 2], math.sqrt(1.0 - s * s)
    out.gates[i] = cg.Gate(cg.U1, out.gates[i].q0, u=(c, 0.0, -s, 0.0, s, 0.0, c, 0.0), cycle=out.gates[i].cycle)
    return out


def worst(circ, p, seed):
    """Largest error of four slice terms (the largest ones) against the oracle, and their norm."""
    x = cg.random_bitstrings(circ.n_qubits, 1, seed + 1)[0]
    terms = p.slice_terms([x]).cpu().numpy()[0].astype(np.complex128)
    ids = np.argsort(-np.abs(terms))[:4]
    ref = VE.slice_terms(circ, x, p.order, p.slices, slice_ids=ids)
    return np.linalg.norm(terms[ids] - ref), np.linalg.norm(ref)


@pytest.mark.parametrize("args,there", CASES)
def test_forms_vs_oracle(args, there):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    circ = cg.grid_circuit(*args[:4])
    p = plan(circ, args)
    got = launched(p.image(), 2)
    assert set(there) <= got, got
    err, size = worst(circ, p, args[3])
    # at most 8.5 truncations of half of 2^-23 a launch, all in one direction, and 2^-20 for the
    # roundings of the program's other sums
    assert err <= (8.5 * 2.0 ** -24 * len(pairs_of(p.image())) + 8.5 * 2.0 ** -24 * p.info["n_gemm_steps"] + 2.0 ** -20) * size
    # one gate's entries in the ratio 30: three parts, no merged steps
    other = unequal(circ, 1.0 / 30.0)
    p = plan(other, args, order=p.order, slices=p.slices)
    assert len(pairs_of(p.image())) + len(reduces_of(p.image())) == 0
    THREE_PARTS.update(launched(p.image(), 3))
    err, _ = worst(other, p, args[3])
    assert err < 1e-5 * 2.0 ** (-circ.n_qubits / 2)


def test_three_part_forms_were_all_launched():
    assert {(nt, form) for _, nt, form, _ in THREE_PARTS} >= {(nt, form) for nt in (16, 32, 64, 128, 256) for form in (S, B)}
