"""The work that users of this framework have it do, as cases to measure.

Every case evaluates the Jamiolkowski fidelity F_J of noisy circuits through the C-ABI mirrors in
paper_2103_11595_gb300/ajf.py. A case fixes the circuits' structure (family, sizes, gate and noise
places: `layout`) and how they are evaluated; the seed of `prepare` draws the values (gate angles
and matrices, noise strengths), which is what changes from call to call in a user's program.
"""
import functools
import math

import numpy as np
import torch

from paper_2103_11595_gb300 import ajf
from paper_2103_11595_gb300 import workloads as W

# family  tiny: gates from {H, T, S, CX, Rz}, depolarising noises (the small-network workload)
#         line: U3 layers and nearest-neighbour CX bricks, mixed noises (the mid workload)
#         dep:  the same circuits with depolarising noises only (the batching workload)
#         grid: brickwork of Haar SU(4) on a rows x cols grid, a depolarising channel on both qubits
#               of every gate (the precision workload); `gates` is its depth, `n` rows * cols
# how     single:     one fidelity call (and the traces of an F64 Alg. I call)
#         batch:      one ajf_fidelity_batch call over `count` circuits, each on its own stream
#         persistent: one ajf_launch_persistent call over `count` small networks
#         sliced:     one fidelity call of a plan with 3 sliced bonds (a tight memory budget)
#         reload:     new gate and noise values: load, plan (known structure), one fidelity call
EPS = 0.05
GRID = {6: (2, 3), 9: (3, 3), 12: (3, 4), 16: (4, 4), 20: (4, 5)}


def listed():
    def c(name, family, n, gates, noises, alg, precision, how, count, layout, graph):
        return {"name": name, "family": family, "n": n, "gates": gates, "noises": noises, "alg": alg,
                "precision": precision, "how": how, "count": count, "layout": layout, "graph": graph}

    return [
        # the smallest call: one 3-qubit circuit checked with the default options, all traces wanted
        c("tiny_alg1_f64", "tiny", 3, 20, 2, 1, "f64", "single", 1, 0, False),
        # a test suite's worth of small circuits in one launch
        c("tiny100_persistent", "tiny", 3, 20, 2, 2, "f64", "persistent", 100, 0, False),
        # an ordinary circuit with the default options, every Kraus combination's trace
        c("line10_alg1_f64", "dep", 10, 110, 6, 1, "f64", "single", 1, 3, False),
        # the headline circuit with the default options (FP64): the largest work in FP64
        c("line16_alg2_f64", "line", 16, 200, 10, 2, "f64", "single", 1, 1, False),
        # a shallow 2-D circuit with noise after every gate, default options
        c("grid20_alg2_f64", "grid", 20, 4, 0, 2, "f64", "single", 1, 0, False),
        # the headline circuit evaluated again and again in the FP32-class tensor-core mode
        c("line16_alg2_bf16x6", "line", 16, 200, 10, 2, "bf16x6", "single", 1, 1, True),
        # the same on CUDA cores' FP32 mode
        c("line16_alg2_f32", "line", 16, 200, 10, 2, "f32", "single", 1, 2, True),
        # the 2-D circuit in the fastest split mode
        c("grid20_alg2_bf16x3", "grid", 20, 4, 0, 2, "bf16x3", "single", 1, 1, True),
        # the benchmark's batch: ten headline circuits at once
        c("line16_batch10_bf16x6", "line", 16, 200, 10, 2, "bf16x6", "batch", 10, 0, True),
        # twelve circuits of uneven odd sizes (n from 8 up), 4096 Kraus combinations each
        c("uneven_batch12_alg1_bf16x6", "dep", 8, 90, 6, 1, "bf16x6", "batch", 12, 5, True),
        # the headline circuit under a memory budget: 2^3 bond slices
        c("line16_sliced_bf16x6", "line", 16, 200, 10, 2, "bf16x6", "sliced", 1, 3, True),
        # a parameter scan: the same circuit structure with new values on every call
        c("line16_reload_bf16x6", "line", 16, 200, 10, 2, "bf16x6", "reload", 1, 4, True),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    layout = rng.randrange(10, 10 ** 6)
    family = rng.choice(["tiny", "line", "line", "line", "dep", "dep", "grid"])
    precision = rng.choice(["f64", "f64", "f64", "bf16x6", "bf16x6", "bf16x6", "f32", "tf32x3", "bf16x3", "f16x3"])
    graph = rng.random() < 0.5
    if family == "tiny":
        how, count = rng.choice([("single", 1), ("persistent", spread(2, 200))])
        return {"family": family, "n": rng.randint(2, 5), "gates": spread(8, 40), "noises": rng.randint(1, 3),
                "alg": rng.choice([1, 2]), "precision": "f64", "how": how, "count": count, "layout": layout,
                "graph": graph and how == "single"}
    if family == "grid":
        return {"family": family, "n": rng.choice(sorted(GRID)), "gates": rng.randint(2, 4), "noises": 0, "alg": 2,
                "precision": precision, "how": rng.choice(["single", "reload"]), "count": 1, "layout": layout,
                "graph": graph}
    if family == "dep":
        how, count = rng.choice([("single", 1), ("batch", rng.randint(2, 12)), ("reload", 1)])
        n = rng.randint(4, 10) if how == "batch" else rng.randint(4, 12)
        return {"family": family, "n": n, "gates": spread(3 * n, 10 * n), "noises": rng.randint(1, 6), "alg": 1,
                "precision": precision, "how": how, "count": count, "layout": layout, "graph": graph}
    how = rng.choice(["single", "single", "batch", "sliced", "reload"])
    n = rng.randint(5, 15 if precision == "f64" and how == "single" else 10 if precision == "f64" else 16)
    return {"family": family, "n": n, "gates": spread(4 * n, 12 * n), "noises": rng.randint(1, 10), "alg": 2,
            "precision": precision, "how": how, "count": rng.randint(2, 8) if how == "batch" else 1,
            "layout": layout, "graph": graph}


# ------------------------------------------------------------------ circuits


def _u3(t, f, l):
    c, s = math.cos(t / 2), math.sin(t / 2)
    return np.array([[c, -np.exp(1j * l) * s], [np.exp(1j * f) * s, np.exp(1j * (f + l)) * c]])


def _haar(r, d):
    q, u = np.linalg.qr(r.standard_normal((d, d)) + 1j * r.standard_normal((d, d)))
    return q * (np.diag(u) / np.abs(np.diag(u)))


def _kraus(r, kind):
    if kind == "dep":  # error probability p
        p = r.uniform(1e-4, 1e-2)
        x, z = np.array([[0, 1], [1, 0]]), np.diag([1, -1])
        return np.stack([math.sqrt(1 - 0.75 * p) * np.eye(2), math.sqrt(p / 4) * x, math.sqrt(p / 4) * 1j * (x @ z),
                         math.sqrt(p / 4) * z]).astype(complex)
    g = r.uniform(1e-4, 1e-2)  # amplitude damping
    return np.array([[[1, 0], [0, math.sqrt(1 - g)]], [[0, math.sqrt(g)], [0, 0]]], dtype=complex)


def _circuit(case, which, seed):
    """(n, gates [(qubits, matrix)], noises [(after gate, qubits, Kraus stack)]) of circuit `which`: the
    structure from the case's layout, the values from the seed."""
    lay = np.random.default_rng([case["layout"], which])
    val = np.random.default_rng([seed, which])
    fam, n, ng = case["family"], case["n"], case["gates"]
    gates, places = [], []
    cx = np.eye(4)[[0, 1, 3, 2]].astype(complex)
    if fam == "grid":
        rows, cols = GRID[n]
        at = lambda r, c: r * cols + c  # noqa: E731
        colours = [[(at(r, c), at(r, c + 1)) for r in range(rows) for c in range(o, cols - 1, 2)] for o in (0, 1)]
        colours += [[(at(r, c), at(r + 1, c)) for r in range(o, rows - 1, 2) for c in range(cols)] for o in (0, 1)]
        for d in range(ng):
            for pair in colours[d % 4]:
                gates.append((pair, _haar(val, 4)))
                places += [(len(gates) - 1, q, "dep") for q in pair]
    elif fam == "tiny":
        fixed = [np.array([[1, 1], [1, -1]]) / math.sqrt(2), np.diag([1, np.exp(0.25j * math.pi)]), np.diag([1, 1j])]
        for _ in range(ng):
            k = int(lay.integers(5))
            if k == 3:
                a, b = lay.choice(n, size=2, replace=False)
                gates.append(((int(a), int(b)), cx))
            else:
                t = val.uniform(0, 2 * math.pi)
                m = np.diag([np.exp(-0.5j * t), np.exp(0.5j * t)]) if k == 4 else fixed[k]
                gates.append(((int(lay.integers(n)),), m.astype(complex)))
    else:
        if case["how"] == "batch" and fam == "dep":  # uneven sizes
            n, ng = n + (2 * which + 1) % 9 % (n + 1), ng + 13 * which
        layer = 0
        while len(gates) < ng:
            if layer % 2 == 0:
                gates += [((q,), _u3(*val.uniform(0, 2 * math.pi, size=3))) for q in range(n)]
            else:
                gates += [((q, q + 1), cx) for q in range(layer // 2 % 2, n - 1, 2)]
            layer += 1
        gates = gates[:ng]
    if fam != "grid":
        for g in sorted(lay.choice(len(gates), size=min(case["noises"], len(gates)), replace=False).tolist()):
            qs = gates[g][0]
            kind = "dep" if fam != "line" or lay.random() < 0.5 else "ad"
            places.append((g, qs[int(lay.integers(len(qs)))], kind))
    return n, gates, [(g, (q,), _kraus(val, kind)) for g, q, kind in places]


def _instance(case, which, seed):
    n, gates, noises = _circuit(case, which, seed)
    return W.Instance(n, [W.Gate(q, m) for q, m in gates], [W.Noise(g, q, k) for g, q, k in noises])


# ------------------------------------------------------------------ one pass


def _plan(handle, case):
    return ajf.ajf_plan(handle, case["alg"], precision=case["precision"], use_graph=case["graph"],
                        lowering="persistent" if case["how"] == "persistent" else "default",
                        slice_bonds=3 if case["how"] == "sliced" else 0)


def prepare(case, seed):
    """Contexts with the circuits loaded and planned; for `reload` also the packed values of new calls."""
    ctxs = []
    for k in range(case["count"]):
        ctx = ajf.Context(torch.cuda.current_device())
        ajf.load_instance(ctx.handle, _instance(case, k, seed))
        _plan(ctx.handle, case)
        ctxs.append(ctx)
    state = {"case": case, "ctxs": ctxs, "handles": [c.handle for c in ctxs]}
    if case["how"] == "persistent":
        state["results"] = torch.zeros((case["count"], 3), dtype=torch.float64, device="cuda")
        for h in state["handles"]:
            ajf.ajf_upload(h)
        torch.cuda.synchronize()
    elif case["how"] == "reload":
        state["packed"] = ajf.pack_instance(_instance(case, 0, seed))
    elif case["alg"] == 1:
        state["combinations"] = _combinations(case)
    return state


def _combinations(case):
    return math.prod(k.shape[0] for _, _, k in _circuit(case, 0, 0)[2])


def run(state):
    case, handles = state["case"], state["handles"]
    if case["how"] == "persistent":
        ajf.ajf_launch_persistent(handles, state["results"].data_ptr())
        return state["results"]
    if case["how"] == "batch":
        return [_result(r, case) for r in ajf.ajf_fidelity_batch(handles, case["alg"], EPS)]
    h = handles[0]
    if case["how"] == "reload":
        ajf.load_packed(h, state["packed"])
        _plan(h, case)
    out = _result(ajf.ajf_fidelity(h, EPS), case)
    if case["alg"] == 1 and case["precision"] == "f64" and case["how"] == "single":
        out["traces"] = ajf.ajf_alg1_traces(h, state["combinations"])
    return out


def _result(r, case):
    """A call's result as it comes; the FP64 mode's numbers are kept as FP64."""
    return {k: np.float64(v) if case["precision"] == "f64" and isinstance(v, float) else v for k, v in r.items()}


# ------------------------------------------------------------------ work


@functools.lru_cache(maxsize=None)
def _flops(key, which):
    case = dict(key)
    with ajf.Context(-1) as ctx:  # a host-only context: the pairwise contractions' multiply-adds
        ajf.load_instance(ctx.handle, _instance(case, which, 0))
        return ajf.ajf_plan(ctx.handle, case["alg"], precision=case["precision"])["flops"]


def work(case):
    """Gate and Kraus matrices in, results (and traces) out; 8 flops per complex multiply-add of the
    contraction order that the planner finds for the whole network."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    nbytes = flops = 0
    for k in range(case["count"]):
        _, gates, noises = _circuit(case, k, 0)
        nbytes += 16 * (sum(m.size for _, m in gates) + sum(x.size for _, _, x in noises)) + 24
        flops += _flops(key, k)
    if case["alg"] == 1 and case["precision"] == "f64" and case["how"] == "single":
        nbytes += 16 * _combinations(case)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ 64-bit values


def _closed(n, gates, noises):
    """The closed sequence E then U^dagger as [(qubits, matrix or Kraus stack, gate index or None)],
    without the gates that cancel against their own adjoints inside the trace."""
    seq, by_gate = [], {}
    for g, q, k in noises:
        by_gate.setdefault(g, []).append((q, k, None))
    for g, (q, m) in enumerate(gates):
        seq.append((q, m, g))
        seq += by_gate.get(g, [])
    seq += [(q, m.conj().T, g) for g, (q, m) in reversed(list(enumerate(gates)))]
    changed = True
    while changed:
        changed = False
        for i, (q, _, g) in enumerate(seq):
            j = next((j for j in range(i + 1, len(seq)) if g is not None and seq[j][2] == g), None)
            if j is None:
                continue
            for between in (seq[i + 1:j], seq[j + 1:] + seq[:i]):
                if not any(set(q) & set(x[0]) for x in between):
                    del seq[j], seq[i]
                    changed = True
                    break
            if changed:
                break
    return seq


def _network(n, seq, doubled):
    """Tensors (array, labels) of the closed network, its open labels, and the wires nothing touches."""
    fresh = iter(range(10 ** 9))
    first = [[next(fresh) for _ in range(n)] for _ in range(2)]
    wires = [list(w) for w in first]
    tensors, opens = [], []

    def put(m, q, side, extra=None):
        a = len(q)
        new = [next(fresh) for _ in q]
        t = m.reshape((m.shape[0],) * (extra is not None) + (2,) * (2 * a))
        tensors.append([t, ([extra] if extra is not None else []) + new + [wires[side][x] for x in q]])
        for x, y in zip(q, new):
            wires[side][x] = y

    for q, m, g in seq:
        extra = None
        if g is None:
            extra = next(fresh)
            if not doubled:
                opens.append(extra)
        put(m, q, 0, extra)
        if doubled:
            put(m.conj(), q, 1, extra)
    loops = 0
    for side in range(2 if doubled else 1):
        for x in range(n):
            if wires[side][x] == first[side][x]:
                loops += 1
            else:  # join the output to the input through an identity
                tensors.append([np.eye(2, dtype=complex), [wires[side][x], first[side][x]]])
    return tensors, opens, loops


def _contract(tensors, opens):
    """Pairwise contraction, cheapest growth first, complex128."""
    dims = {l: t.shape[i] for t, ls in tensors for i, l in enumerate(ls)}
    size = lambda ls: math.prod(dims[l] for l in ls)  # noqa: E731
    live = dict(enumerate(tensors))
    top = len(live)
    while len(live) > 1:
        where, best = {}, None
        for i, (_, ls) in live.items():
            for l in ls:
                where.setdefault(l, []).append(i)
        for i, j in {tuple(v) for v in where.values() if len(v) == 2}:
            a, b = live[i][1], live[j][1]
            out = set(a) ^ set(b)
            cost = (size(out) - size(a) - size(b), size(out), i, j)
            if best is None or cost < best:
                best = cost
        i, j = best[2:] if best else sorted(live, key=lambda k: live[k][0].size)[:2]
        (x, a), (y, b) = live.pop(i), live.pop(j)
        shared = [l for l in a if l in b]
        live[top] = [np.tensordot(x, y, ([a.index(l) for l in shared], [b.index(l) for l in shared])),
                     [l for l in a if l not in shared] + [l for l in b if l not in shared]]
        top += 1
    (x, labels), = live.values()
    return x.transpose([labels.index(l) for l in opens])


def exact(case, seed):
    outs = []
    for k in range(case["count"]):
        n, gates, noises = _circuit(case, k, seed)
        seq = _closed(n, gates, noises)
        traces = None
        if case["alg"] == 1:
            tensors, opens, loops = _network(n, seq, False)
            traces = (_contract(tensors, opens) * 2.0 ** loops).reshape(-1)
            s = math.fsum((traces * traces.conj()).real.tolist())
        else:
            tensors, _, loops = _network(n, seq, True)
            s = float(_contract(tensors, []).real) * 2.0 ** loops
        d2 = 4.0 ** n
        outs.append({"F": np.float64(s / d2), "one_minus_F": np.float64((d2 - s) / d2), "S": np.float64(s),
                     "traces_done": None, "equivalent": None})
    if case["how"] == "persistent":
        return np.array([[o["S"], o["F"], o["one_minus_F"]] for o in outs])
    if case["how"] == "batch":
        return outs
    if case["alg"] == 1 and case["precision"] == "f64" and case["how"] == "single":
        outs[0]["traces"] = traces
    return outs[0]
