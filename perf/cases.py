"""The workloads this framework is timed on, and their results in 64 bits.

Each case is a call that a program makes of the public interface: amplitudes <x|C|0> and
slice terms of random grid circuits, and amplitudes with the derivatives of rotation
circuits. Sizes are those of the repository's benchmark workloads and tests.
"""
import json
import math
import os

import numpy as np
import torch

import circuitgen as cg
import paper_1805_01450_gb300 as qvx
from paper_1805_01450_gb300 import autograd as qvx_autograd

DEVICE = "cuda"
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# keyword arguments of Plan that a case may hold under the same name
PLAN_KEYS = ("n_slices", "inner_slices", "engine", "warps_per_item", "host_merge_rank", "plan_trials", "tensor_cores",
             "mem_budget_bytes", "gradient")


def listed():
    fused = dict(n_slices=12, inner_slices=5, warps_per_item=16, host_merge_rank=10, plan_trials=64)
    gib = 1 << 30
    return [
        # the smallest call: one amplitude of a 16-qubit circuit, the bitstring a Python integer
        dict(name="grid4x4d10", call="amplitude", rows=4, cols=4, depth=10, circuit=1001, batch=1, n_slices=0),
        # one amplitude of a 36-qubit circuit in a loop that keeps its buffers (the latency-bound
        # on-chip engine with 12 sliced variables)
        dict(name="grid6x6d25", call="amplitude_loop", rows=6, cols=6, depth=25, circuit=2001, batch=1, **fused),
        # the same amplitude from page-locked host memory into page-locked host memory
        dict(name="grid6x6d25-host", call="amplitude_host", rows=6, cols=6, depth=25, circuit=2001, batch=1, **fused),
        # 64 amplitudes of that circuit per call: the on-chip engine with every SM busy
        dict(name="grid6x6d25-b64", call="amplitude_loop", rows=6, cols=6, depth=25, circuit=2001, batch=64,
             **dict(fused, warps_per_item=4)),
        # 1024 amplitudes of a 49-qubit circuit (output statistics, fidelity estimates)
        dict(name="grid7x7d30-b1024", call="amplitude_loop", rows=7, cols=7, depth=30, circuit=3001, batch=1024,
             n_slices=2, inner_slices=2, engine="stepwise", plan_trials=64, mem_budget_bytes=32 * gib),
        # a few amplitudes of that circuit with the planner's default engine
        dict(name="grid7x7d30-default", call="amplitude", rows=7, cols=7, depth=30, circuit=3001, batch=16, n_slices=8),
        # one training step of a 25-qubit rotation circuit: |alpha|^2 and its gradient in all
        # 1000 angles through torch.autograd (forward and backward)
        dict(name="rot5x5d20-train", call="train", rows=5, cols=5, depth=20, circuit=4001, batch=1, n_slices=8,
             inner_slices=1, gradient=True),
        # amplitudes and Jacobian of a batch of bitstrings
        dict(name="rot5x5d20-jacobian-b16", call="jacobian", rows=5, cols=5, depth=20, circuit=4001, batch=16, n_slices=8,
             inner_slices=1, gradient=True),
        # every slice term of 42-qubit amplitudes with the dense contractions on the tensor cores
        dict(name="grid6x7d40-terms", call="terms", rows=6, cols=7, depth=40, circuit=2, batch=2, n_slices=10,
             inner_slices=5, engine="stepwise", tensor_cores=True, plan_trials=16),
        # every slice term of a 64-qubit depth-40 amplitude (amplitude() adds exactly these):
        # the three circuits with recorded orderings
        dict(name="grid8x8d40-s5001", call="terms", rows=8, cols=8, depth=40, circuit=5001, batch=1, recorded=True),
        dict(name="grid8x8d40-s5002", call="terms", rows=8, cols=8, depth=40, circuit=5002, batch=1, recorded=True),
        dict(name="grid8x8d40-s5003", call="terms", rows=8, cols=8, depth=40, circuit=5003, batch=1, recorded=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: grids from 2 x 2 to 8 x 8, batches spread over
    their logarithm, other circuits, slice counts and parts of the slice range."""
    kind = rng.choice(("amplitude", "on-chip", "batch", "default", "gradient", "terms", "recorded"))
    seed = rng.randrange(1, 100000)
    if kind == "amplitude":
        return dict(call="amplitude", rows=rng.randint(2, 4), cols=rng.randint(2, 5), depth=rng.randint(4, 16), circuit=seed,
                    batch=_log(rng, 1, 16), n_slices=rng.randint(0, 3))
    if kind == "on-chip":
        k = rng.randint(10, 12)
        return dict(call=rng.choice(("amplitude_loop", "amplitude_host")), rows=rng.randint(5, 6), cols=6,
                    depth=rng.randint(16, 25), circuit=seed, batch=_log(rng, 1, 100), n_slices=k,
                    inner_slices=rng.randint(3, 5), warps_per_item=rng.choice((2, 4, 8, 16)), host_merge_rank=8,
                    plan_trials=16)
    if kind == "batch":
        return dict(call="amplitude_loop", rows=rng.randint(6, 7), cols=7, depth=rng.randint(20, 28), circuit=seed,
                    batch=_log(rng, 16, 700), n_slices=3, inner_slices=rng.randint(0, 3), engine="stepwise",
                    plan_trials=16, mem_budget_bytes=16 << 30)
    if kind == "default":
        return dict(call="amplitude", rows=rng.randint(6, 7), cols=rng.randint(6, 7), depth=rng.randint(24, 30), circuit=seed,
                    batch=_log(rng, 1, 16), n_slices=8)
    if kind == "gradient":
        return dict(call=rng.choice(("train", "jacobian")), rows=rng.randint(3, 5), cols=rng.randint(3, 5),
                    depth=rng.randint(6, 20), circuit=seed, batch=_log(rng, 1, 16), n_slices=rng.randint(6, 8), inner_slices=1,
                    gradient=True)
    if kind == "terms":
        return dict(call="terms", rows=6, cols=rng.randint(5, 7), depth=rng.randint(32, 40), circuit=seed,
                    batch=rng.randint(1, 3), n_slices=10, inner_slices=rng.randint(3, 5), engine="stepwise",
                    tensor_cores=True, plan_trials=16)
    first = rng.randrange(0, 1024)
    return dict(call="terms", rows=8, cols=8, depth=40, circuit=rng.choice((5001, 5002, 5003)), batch=1, recorded=True,
                first=first, count=max(1, _log(rng, 32, 1024) * (1024 - first) // 1024))


def _circuit(case):
    make = cg.rotation_circuit if case.get("gradient") else cg.grid_circuit
    return make(case["rows"], case["cols"], case["depth"], case["circuit"])


def _ordering(case):
    with open(os.path.join(ROOT, "paper_1805_01450_gb300", "orderings", "grid8x8d40-s%d.json" % case["circuit"])) as f:
        return json.load(f)


def _plan(case, circ):
    if case.get("recorded"):   # the variant that the benchmark keeps for this circuit
        d = _ordering(case)
        return qvx.Plan(circ, order=d["order"], slices=d["slices"], inner_slices=d["variant"]["inner_slices"],
                        engine="stepwise", tensor_cores=True, mem_budget_bytes=64 << 30)
    return qvx.Plan(circ, **{k: case[k] for k in PLAN_KEYS if k in case})


def _inputs(case, seed):
    """(bitstrings as Python integers, angles or None), from the seed alone."""
    n = case["rows"] * case["cols"]
    rng = np.random.default_rng(seed)
    xs = [int.from_bytes(rng.bytes(16), "little") & ((1 << n) - 1) for _ in range(case["batch"])]
    n_angles = 2 * n * case["depth"]
    return xs, rng.uniform(0.0, 2.0 * math.pi, n_angles) if case.get("gradient") else None


def prepare(case, seed):
    circ = _circuit(case)
    plan = _plan(case, circ)
    xs, thetas = _inputs(case, seed)
    state = {"case": case, "plan": plan, "xs": xs}
    words = torch.tensor(qvx.bitstring_words(xs, plan.words), dtype=torch.int64)
    if case["call"] == "amplitude_host":
        state["bits"] = words.pin_memory()
        state["out"] = torch.empty(2 * len(xs), dtype=torch.float64).pin_memory()
    else:
        state["bits"] = words.to(DEVICE)
    if thetas is not None:
        state["thetas"] = torch.tensor(thetas, dtype=torch.float64, device=DEVICE)
    if case["call"] == "amplitude_loop":
        state["out"] = torch.empty(2 * len(xs), dtype=torch.float64, device=DEVICE)
    state["ws"] = plan.workspace(len(xs))
    return state


def run(state):
    case, plan = state["case"], state["plan"]
    call = case["call"]
    if call == "amplitude":          # Python integers in, a device tensor out
        return plan.amplitude(state["xs"], workspace=state["ws"])
    if call == "amplitude_loop":     # the program checked its bitstrings and keeps its buffers
        return plan.amplitude(state["bits"], workspace=state["ws"], out=state["out"], validate=False)
    if call == "amplitude_host":
        return plan.amplitude_host(state["bits"], out=state["out"], workspace=state["ws"])
    if call == "terms":
        first = case.get("first", 0)
        return plan.slice_terms(state["bits"], slice_begin=first, slice_count=case.get("count"), workspace=state["ws"])
    if call == "jacobian":
        return plan.amplitude_grad(state["bits"], state["thetas"], workspace=state["ws"])
    thetas = state["thetas"].detach().requires_grad_()
    alpha = qvx_autograd.amplitude(plan, state["bits"], thetas)
    loss = (alpha.abs() ** 2).sum()
    loss.backward()
    return {"alpha": alpha.detach(), "loss": loss.detach(), "grad": thetas.grad}


def work(case):
    """Real flops of the elimination (8 per complex multiply-add) over the slice terms of the
    call, and the bytes of its inputs and outputs; tensors in between need not touch memory."""
    circ = _circuit(case)
    info = _plan(case, circ).info
    n = case["rows"] * case["cols"]
    batch = case["batch"]
    flops = info["grad_flops_per_amplitude"] if case.get("gradient") else info["flops_per_amplitude"]
    terms = 1 << info["n_sliced"]
    part = case.get("count", terms) / terms
    gates = 64 * len(circ.gates)
    out = 8 * terms * part if case["call"] == "terms" else 16
    if case.get("gradient"):
        out += 16 * info["n_params"] if case["call"] == "jacobian" else 8 * info["n_params"]
    return {"bytes": gates + batch * (8 * ((n + 63) // 64) + out), "flops": batch * flops * part}


# ---------------------------------------------------------------- results in 64 bits
_R2 = 1.0 / math.sqrt(2.0)
_SINGLE = {cg.H: [[_R2, _R2], [_R2, -_R2]],
           cg.SQRT_X: [[0.5 + 0.5j, 0.5 - 0.5j], [0.5 - 0.5j, 0.5 + 0.5j]],
           cg.SQRT_Y: [[0.5 + 0.5j, -0.5 - 0.5j], [0.5 + 0.5j, 0.5 + 0.5j]]}
_T = [1.0, complex(math.cos(math.pi / 4), math.sin(math.pi / 4))]
_BATCH = -1   # mode of the bitstrings in the contraction


def _network(circ, xs):
    """Tensors (modes, complex128 CUDA array) of the circuit's graph with inputs 0 and the
    outputs fixed to the bitstrings; variable ids run in order of (qubit, gate on the qubit)."""
    n = circ.n_qubits
    count = [sum(1 for g in circ.gates if g.q0 == q and g.kind not in (cg.CZ, cg.T)) for q in range(n)]
    first = np.concatenate([[0], np.cumsum([max(c - 1, 0) for c in count])])
    done = [0] * n
    bit = {q: torch.tensor([(x >> q) & 1 for x in xs], device=DEVICE) for q in range(n)}

    def place(q, k):   # the value of qubit q after its k-th non-diagonal gate
        if k == 0:
            return "zero"
        return ("out", q) if k == count[q] else int(first[q]) + k - 1

    def tensor(places, data):
        data = torch.tensor(data, dtype=torch.complex128, device=DEVICE)
        for axis, p in reversed(list(enumerate(places))):
            if p == "zero":
                data = data.select(axis, 0)
        places = [p for p in places if p != "zero"]
        outs = [a for a, p in enumerate(places) if isinstance(p, tuple)]
        if outs:   # fixed outputs become one leading axis over the bitstrings
            index = tuple(bit[p[1]] if isinstance(p, tuple) else slice(None) for p in places)
            order = outs + [a for a in range(len(places)) if a not in outs]
            data = data.permute(order)
            data = data[tuple(index[a] for a in outs)]
            modes = [_BATCH] + [places[a] for a in range(len(places)) if a not in outs]
        else:
            modes = list(places)
        return modes, data

    out = []
    for g in circ.gates:
        if g.kind == cg.CZ:
            out.append(tensor([place(g.q0, done[g.q0]), place(g.q1, done[g.q1])], [[1, 1], [1, -1]]))
        elif g.kind == cg.T:
            out.append(tensor([place(g.q0, done[g.q0])], _T))
        else:
            done[g.q0] += 1
            out.append(tensor([place(g.q0, done[g.q0]), place(g.q0, done[g.q0] - 1)], _SINGLE[g.kind]))
    if any(c == 0 for c in count):
        raise ValueError("a qubit without a non-diagonal gate")
    return out


def _product(a, b, keep):
    """Contraction of two tensors, summed over the modes outside `keep`."""
    modes = list(dict.fromkeys(a[0] + b[0]))
    name = {m: i for i, m in enumerate(modes)}
    out = [m for m in modes if m in keep]
    return out, torch.einsum(a[1], [name[m] for m in a[0]], b[1], [name[m] for m in b[0]], [name[m] for m in out])


def _eliminate(tensors, order, open_modes):
    """Bucket elimination in the given order; the result over the open modes in their order."""
    live = [t for t in tensors if t[0]]
    scalar = 1.0
    for t in tensors:
        if not t[0]:
            scalar = scalar * t[1]

    def merge(group):
        nonlocal live
        others = {m for t in live if not any(t is u for u in group) for m in t[0]}
        live = [t for t in live if not any(t is u for u in group)]
        group = list(group)
        while len(group) > 1:
            pairs = [(len(set(p[0]) | set(r[0])), i, j) for i, p in enumerate(group) for j, r in enumerate(group) if i < j]
            _, i, j = min(pairs)
            a, b = group[i], group[j]
            group = [t for k, t in enumerate(group) if k not in (i, j)]
            keep = others | open_set | {m for t in group for m in t[0]}
            group.append(_product(a, b, keep))
        return group[0]

    open_set = set(open_modes)
    for v in order:
        group = [t for t in live if v in t[0]]
        if not group:
            continue
        modes, data = merge(group)
        if v in modes:   # a variable of one tensor alone
            data = data.sum(modes.index(v))
            modes = [m for m in modes if m != v]
        live.append((modes, data))
    modes, data = merge(list(live)) if live else ([], torch.ones((), dtype=torch.complex128, device=DEVICE))
    present = [m for m in open_modes if m in modes]
    data = data.permute([modes.index(m) for m in present])
    for i, m in enumerate(open_modes):
        if m not in present:
            data = data.unsqueeze(i)
    return data * scalar


def _terms64(case, circ, plan, xs, first, count):
    """Slice terms first ... first + count - 1 of every bitstring; slice number s gives sliced
    variable i the value of bit i of s. The low variables stay open, the others are looped."""
    net = _network(circ, xs)
    k = len(plan.slices)
    inner = min(k, int(plan.info["n_inner"]))
    low, high = plan.slices[:inner], plan.slices[inner:]
    out = torch.empty(len(xs), count, dtype=torch.complex128, device=DEVICE)
    for o in range(first >> inner, ((first + count - 1) >> inner) + 1):
        value = {v: (o >> i) & 1 for i, v in enumerate(high)}
        tensors = []
        for modes, data in net:
            for axis in reversed(range(len(modes))):
                if modes[axis] in value:
                    data = data.select(axis, value[modes[axis]])
            tensors.append(([m for m in modes if m not in value], data))
        # open modes: bitstrings slowest, then the open variables from high to low
        t = _eliminate(tensors, plan.order, [_BATCH] + low[::-1]).expand(len(xs), *([2] * inner)).reshape(len(xs), -1)
        s0 = max(first, o << inner)
        s1 = min(first + count, (o + 1) << inner)
        out[:, s0 - first:s1 - first] = t[:, s0 - (o << inner):s1 - (o << inner)]
    return out


def _apply(psi, m, q, n):
    """2 x 2 matrix on qubit q of states [batch, 2^n] (bit q of the index is qubit q)."""
    v = psi.view(-1, 1 << (n - 1 - q), 2, 1 << q)
    return torch.stack((m[0][0] * v[:, :, 0] + m[0][1] * v[:, :, 1], m[1][0] * v[:, :, 0] + m[1][1] * v[:, :, 1]),
                       2).view(psi.shape)


def _gradients64(circ, xs, thetas):
    """(alpha [batch], d alpha / d theta [batch, angles]) by the state vector: forward, then
    the costate <x| swept back through the gates."""
    n = circ.n_qubits
    index = torch.arange(1 << n, device=DEVICE)
    psi = torch.zeros(1, 1 << n, dtype=torch.complex128, device=DEVICE)
    psi[0, 0] = 1.0

    def rotation(g):
        t, e = thetas[g.param] / 2, complex(math.cos(g.phi), math.sin(g.phi))
        c, s = math.cos(t), math.sin(t)
        u = [[c, -1j * s * e.conjugate()], [-1j * s * e, c]]
        d = [[-s / 2, -0.5j * c * e.conjugate()], [-0.5j * c * e, -s / 2]]
        return u, d

    def sign(g):
        return 1.0 - 2.0 * ((index >> g.q0) & (index >> g.q1) & 1).to(torch.float64)

    for g in circ.gates:
        psi = psi * sign(g) if g.kind == cg.CZ else _apply(psi, rotation(g)[0], g.q0, n)
    alpha = psi[0, torch.tensor(xs, device=DEVICE)].clone()
    bra = torch.zeros(len(xs), 1 << n, dtype=torch.complex128, device=DEVICE)
    bra[torch.arange(len(xs), device=DEVICE), torch.tensor(xs, device=DEVICE)] = 1.0
    grad = torch.zeros(len(xs), len(thetas), dtype=torch.complex128, device=DEVICE)
    for g in reversed(circ.gates):
        if g.kind == cg.CZ:
            f = sign(g)
            psi, bra = psi * f, bra * f
            continue
        u, d = rotation(g)
        psi = _apply(psi, [[complex(u[j][i]).conjugate() for j in range(2)] for i in range(2)], g.q0, n)
        p = psi.view(1, 1 << (n - 1 - g.q0), 2, 1 << g.q0)
        b = bra.view(len(xs), 1 << (n - 1 - g.q0), 2, 1 << g.q0)
        for i in range(2):
            for j in range(2):   # sum of bra[.., i, ..] d[i][j] psi[.., j, ..]
                left = b[:, :, i].reshape(len(xs), -1)
                grad[:, g.param] += d[i][j] * (left @ p[:, :, j].reshape(-1))
        bra = _apply(bra, [[u[j][i] for j in range(2)] for i in range(2)], g.q0, n)
    return alpha, grad


def exact(case, seed):
    circ = _circuit(case)
    xs, thetas = _inputs(case, seed)
    if case.get("gradient"):
        if case["batch"] << circ.n_qubits > 1 << 29:
            return None   # costates of this batch take too long
        alpha, grad = _gradients64(circ, xs, thetas)
        if case["call"] == "jacobian":
            return alpha, grad
        return {"alpha": alpha, "loss": (alpha.abs() ** 2).sum(), "grad": 2.0 * (alpha.conj()[:, None] * grad).real.sum(0)}
    plan = _plan(case, circ)   # the order and the numbering of the slices that the caller has in hand
    first = case.get("first", 0)
    count = case.get("count") or (1 << len(plan.slices))
    terms = _terms64(case, circ, plan, xs, first, count)
    if case["call"] == "terms":
        return terms
    alpha = terms.sum(1)
    return alpha.cpu().numpy() if case["call"] == "amplitude_host" else alpha
