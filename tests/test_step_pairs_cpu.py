"""Pairs of steps that run as one tensor-core GEMM (StepPair in the device image): for random
operands, the pair's groups and leaf give the consumer's output as the two steps of the program
do, over plans with the leaf on either operand, batch modes taken from a leaf, padded (8) and
long summed indexes."""
import numpy as np
import pytest

import circuitgen as cg
import paper_1805_01450_gb300 as q
from _program_exec import A_LEAF, B_LEAF, GEMM, RUN, Program, _pext

LEAF = np.dtype([("leaf", "<u4"), ("on_rows", "u1"), ("n_b", "u1"), ("n_r", "u1"), ("n_k", "u1"), ("b", RUN, (8,)),
                 ("r", RUN, (8,)), ("k", RUN, (8,))])
PAIR = np.dtype([("producer", "<u4"), ("consumer", "<u4"), ("g", GEMM), ("leaf", LEAF)])
HEAD = 328   # pairs_off and n_pairs follow the fields that Program reads


def pairs_of(image):
    off, n = int(np.frombuffer(image[HEAD:HEAD + 8], "<u8")[0]), int(np.frombuffer(image[HEAD + 8:HEAD + 12], "<u4")[0])
    return np.frombuffer(image[off:off + n * PAIR.itemsize], dtype=PAIR)


def ranks(st):
    return (int(st["a_cb"] + st["nk_ab"] + st["nk_a"]), int(st["b_cb"] + st["nk_ab"] + st["nk_b"]))


def contract(st, a, b):
    """One two-operand step of the program (every summed mode in both operands)."""
    assert st["nk_a"] == 0 and st["nk_b"] == 0
    c = np.arange(1 << int(st["rc"]), dtype=np.int64)
    ia, ib = _pext(c, st["runs_a"], int(st["na_runs"])), _pext(c, st["runs_b"], int(st["nb_runs"]))
    out = np.zeros(c.size, np.complex128)
    for k in range(1 << int(st["nk_ab"])):
        out += a[ia + (k << int(st["a_cb"]))] * b[ib + (k << int(st["b_cb"]))]
    return out


def run_pair(pr, rows, cols, d):
    g, leaf = pr["g"], pr["leaf"]
    nb, nm, nn, nk = (int(g[f]) for f in ("nb", "nm", "nn", "nk"))
    beta, m, n, k = (np.arange(1 << v, dtype=np.int64) for v in (nb, nm, nn, nk))
    mv = lambda idx, f: _pext(idx, g[f], int(g["n_" + f]))
    ld = lambda idx, f: _pext(idx, leaf[f], int(leaf["n_" + f]))
    out = np.zeros(1 << (nb + nm + nn), np.complex128)
    for bb in beta:
        a = rows[mv(bb, "ab") + mv(m, "am")[:, None] + mv(k, "ak")[None, :]]
        b = cols[mv(bb, "bb") + mv(n, "bn")[:, None] + mv(k, "bk")[None, :]]
        f = d[ld(bb, "b") + ld(m if leaf["on_rows"] else n, "r")[:, None] + ld(k, "k")[None, :]]
        c = (a * f) @ b.T if leaf["on_rows"] else a @ (b * f).T
        out[mv(bb, "cb") + mv(m, "cm")[:, None] + mv(n, "cn")[None, :]] = c
    return out


SEEN = {"rows": 0, "cols": 0, "leaf batch": 0, "k8": 0, "long": 0, "swapped": 0}


@pytest.mark.parametrize("r,c_,d,seed,k,inner,trials", [
    (6, 7, 40, 2, 10, 5, 16), (6, 6, 40, 7066, 8, 2, 1), (5, 6, 40, 19, 8, 2, 1), (6, 7, 40, 3, 8, 2, 1),
    (6, 7, 40, 5, 10, 2, 1), (6, 6, 36, 11, 8, 4, 1), (6, 7, 36, 5, 10, 4, 4), (5, 7, 40, 3, 8, 3, 1)])
def test_pairs_equal_their_two_steps(r, c_, d, seed, k, inner, trials):
    p = q.Plan(cg.grid_circuit(r, c_, d, seed), n_slices=k, inner_slices=inner, engine="stepwise", tensor_cores=True,
               plan_trials=trials)
    image = p.image()
    P = Program(image)
    rng = np.random.default_rng(seed)
    rand = lambda rank: rng.standard_normal(1 << rank) + 1j * rng.standard_normal(1 << rank)
    for pr in pairs_of(image):
        s, t = P.steps[int(pr["producer"])], P.steps[int(pr["consumer"])]
        if int(s["rc"]) > 22:
            continue
        a, b = (rand(v) for v in ranks(s))
        x = contract(s, a, b)
        x_is_a = bool(int(t["flags"]) & B_LEAF)
        assert x_is_a != bool(int(t["flags"]) & A_LEAF)
        ra, rb = ranks(t)
        leaf = rand(rb if x_is_a else ra)
        assert x.size == 1 << (ra if x_is_a else rb)
        e = contract(t, x, leaf) if x_is_a else contract(t, leaf, x)
        g = pr["g"]
        # the row operand is the step's A or B: the one at g.a_off
        swap = (int(g["a_off"]), bool(int(g["flags"]) & A_LEAF)) != (int(s["a_off"]), bool(int(s["flags"]) & A_LEAF))
        got = run_pair(pr, b if swap else a, a if swap else b, leaf)
        assert got.size == e.size and int(g["c_off"]) == int(t["c_off"])
        assert np.max(np.abs(got - e)) < 1e-12 * (1 << int(g["nk"])) * np.max(np.abs(leaf)) * 50
        nk = int(g["nk"])
        SEEN["rows" if pr["leaf"]["on_rows"] else "cols"] += 1
        SEEN["leaf batch"] += int(pr["leaf"]["n_b"]) > 0
        SEEN["k8"] += nk == 3
        SEEN["long"] += nk > 7
        SEEN["swapped"] += swap


def test_the_plans_covered_the_forms():
    assert SEEN["rows"] and SEEN["cols"] and SEEN["leaf batch"] and SEEN["swapped"], SEEN
