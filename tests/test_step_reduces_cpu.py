"""Steps merged into the consumer of their result (StepReduce in the device image): the index
maps of the merged form address, for sampled output entries, exactly the operand entries that
the two steps of the program do."""
import os

import numpy as np
import pytest

import circuitgen as cg
import paper_1805_01450_gb300 as q
from _program_exec import A_LEAF, B_LEAF, RUN, Program, _pext

MAPS = ("row_a", "row_d", "row_e", "col_b", "col_d", "col_e", "unit_a", "unit_b", "unit_d", "unit_e", "mo_a", "mo_d", "mo_e",
        "jo_a", "jo_b", "jo_d", "k_a", "k_b")
MAP = np.dtype([("n", "u1"), ("pad", "u1", (3,)), ("runs", RUN, (8,))])
RED = np.dtype([("producer", "<u4"), ("consumer", "<u4"), ("a_off", "<u8"), ("b_off", "<u8"), ("d_off", "<u8"),
                ("e_off", "<u8"), ("flags", "<u4"), ("nk", "u1"), ("nu", "u1"), ("mo", "u1"), ("jo", "u1"), ("jb", "u1"),
                ("jc", "u1"), ("pad", "u1", (2,))] + [(m, MAP) for m in MAPS] + [("tail", "<u4", (1,))])
HEAD = 340   # n_reduces and reduces_off in the program header

PLANS = [(6, 7, 32, 27, 6, 3), (5, 7, 40, 20, 10, 4), (7, 7, 30, 17, 6, 3), (6, 6, 36, 32, 6, 3)]
RECORDED = (5001, 5002)


def reduces_of(image):
    n, off = int(np.frombuffer(image[HEAD:HEAD + 4], "<u4")[0]), int(np.frombuffer(image[HEAD + 4:HEAD + 12], "<u8")[0])
    size = 704
    assert RED.itemsize <= size
    return [np.frombuffer(image[off + i * size:off + i * size + RED.itemsize], dtype=RED)[0] for i in range(n)]


def small_plan(r, c_, d, seed, k, inner):
    return q.Plan(cg.grid_circuit(r, c_, d, seed), n_slices=k, inner_slices=inner, engine="stepwise", tensor_cores=True,
                  order_restarts=2)


def check(p, seed):
    image = p.image()
    P = Program(image)
    reds = reduces_of(image)
    rng = np.random.default_rng(seed)
    for rd in reds:
        s, t = P.steps[int(rd["producer"])], P.steps[int(rd["consumer"])]
        x_is_a = int(t["a_off"]) == int(s["c_off"]) and not int(t["flags"]) & A_LEAF
        xs, dd = ("a", "b") if x_is_a else ("b", "a")
        assert int(rd["e_off"]) == int(t["c_off"]) and int(rd["d_off"]) == int(t[dd + "_off"])
        swap = (int(rd["a_off"]), bool(int(rd["flags"]) & A_LEAF)) != (int(s["a_off"]), bool(int(s["flags"]) & A_LEAF))
        sa, sb = ("b", "a") if swap else ("a", "b")
        mv = lambda name, i: _pext(np.asarray(i, dtype=np.int64), rd[name]["runs"], int(rd[name]["n"]))
        nk, nu, mo, jo, jc, jb = (int(rd[f]) for f in ("nk", "nu", "mo", "jo", "jc", "jb"))
        assert 7 + nu + mo + (7 - jc) == int(t["rc"]) and jo + jc == int(t["nk_ab"]) and nk == int(s["nk_ab"])
        assert 2 <= jc <= 4 and (max(16, 1 << nk) // 16) << jb <= 4
        # k: the same entries of A and B for every summed index of the producer
        k = np.arange(1 << nk)
        assert np.array_equal(mv("k_a", k), k << int(s[sa + "_cb"])) and np.array_equal(mv("k_b", k), k << int(s[sb + "_cb"]))
        seen = set()
        for _ in range(64):
            row, kept, u, m = (int(rng.integers(0, 1 << b)) for b in (7, 7 - jc, nu, mo))
            e = int(mv("row_e", row) + mv("col_e", kept) + mv("unit_e", u) + mv("mo_e", m))
            seen.add(e)
            jj, cc = (v.ravel() for v in np.meshgrid(np.arange(1 << jo), np.arange(1 << jc), indexing="ij"))
            col = (kept << jc) | cc
            got = set(zip((mv("row_a", row) + mv("unit_a", u) + mv("mo_a", m) + mv("jo_a", jj)).tolist(),
                          (mv("col_b", col) + mv("unit_b", u) + mv("jo_b", jj)).tolist(),
                          (mv("row_d", row) + mv("col_d", col) + mv("unit_d", u) + mv("mo_d", m) + mv("jo_d", jj)).tolist()))
            kk = np.arange(1 << int(t["nk_ab"]), dtype=np.int64)
            x = _pext(np.int64(e), t["runs_" + xs], int(t[f"n{xs}_runs"])) + (kk << int(t[xs + "_cb"]))
            d = _pext(np.int64(e), t["runs_" + dd], int(t[f"n{dd}_runs"])) + (kk << int(t[dd + "_cb"]))
            want = set(zip(_pext(x, s["runs_" + sa], int(s[f"n{sa}_runs"])).tolist(),
                           _pext(x, s["runs_" + sb], int(s[f"n{sb}_runs"])).tolist(), d.tolist()))
            assert got == want and len(got) == 1 << int(t["nk_ab"])
        # the groups' maps into E are a permutation of its bits
        bits = [int(mv(f, 1 << i)) for f, n in (("row_e", 7), ("col_e", 7 - jc), ("unit_e", nu), ("mo_e", mo)) for i in range(n)]
        assert sorted(bits) == [1 << i for i in range(int(t["rc"]))]
        # jo bits: the jb highest move B, the others do not
        assert all((int(mv("jo_b", 1 << i)) != 0) == (i >= jo - jb) for i in range(jo))
    return len(reds)


@pytest.mark.parametrize("args", PLANS)
def test_merged_steps_address_the_same_entries(args):
    assert check(small_plan(*args), args[3]) >= 1


@pytest.mark.parametrize("seed", RECORDED)
def test_merged_steps_of_the_recorded_orderings(seed):
    import json
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    with open(os.path.join(root, "paper_1805_01450_gb300", "orderings", f"grid8x8d40-s{seed}.json")) as f:
        d = json.load(f)
    p = q.Plan(cg.grid_circuit(8, 8, 40, seed), order=d["order"], slices=d["slices"],
               inner_slices=d["variant"]["inner_slices"], engine="stepwise", tensor_cores=True, mem_budget_bytes=64 << 30)
    assert check(p, seed) >= 1
