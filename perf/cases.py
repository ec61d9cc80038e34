"""The work that programs have this library do, as cases that can be timed and checked.

A case is a dict of plain values; its "kind" says which public entry point it goes through:
  amplitudes  qfx.amplitudes: x1 batches of a random circuit on a grid (line or tree plan)
  sample      qfx.frugal_sample: amplitudes of x1 batches and the accepted bitstrings
  train       circuit_amplitudes and loss.backward(): gradients of every gate tensor
  batch       qfx.Batch.run: many small items of uneven shapes in one launch
  step        qfx.contract_step: one contraction step in any precision
  permute     qfx.permute: one tensor transpose

Circuits are the library's class of inputs: Hadamards, `depth` cycles of a CZ pattern (eight
patterns cover every edge of the grid once) and one drawn single-qubit gate per qubit,
Hadamards.
"""
import dataclasses
import math
import random

import numpy as np
import torch

import paper_1905_00444_gb300 as qfx

# ------------------------------------------------------------------------------ circuits
H, SQRT_X, SQRT_Y, T, CZ, U1 = 0, 1, 2, 3, 4, 5   # gate kinds of the library's ABI
_R = math.sqrt(0.5)
_MATS = {
    H: np.array([[_R, _R], [_R, -_R]], dtype=np.complex128),
    SQRT_X: 0.5 * np.array([[1 + 1j, 1 - 1j], [1 - 1j, 1 + 1j]]),
    SQRT_Y: 0.5 * np.array([[1 + 1j, -1 - 1j], [1 + 1j, 1 + 1j]]),
    T: np.array([[1, 0], [0, np.exp(0.25j * math.pi)]], dtype=np.complex128),
}
_CZ = np.array([1, 1, 1, -1], dtype=np.complex128)


@dataclasses.dataclass
class Gate:
    layer: int
    q0: int
    q1: int
    kind: int
    mat: np.ndarray


@dataclasses.dataclass
class Grid:
    rows: int
    cols: int
    gates: list


def _pattern(rows, cols, t):
    """Edges of CZ pattern t mod 8: four of horizontal edges, then four of vertical ones."""
    a, b = [(0, 0), (1, 1), (0, 1), (1, 0)][t % 4]
    if t % 8 < 4:
        return [(r * cols + c, r * cols + c + 1) for r in range(rows) for c in range(cols - 1)
                if c % 2 == a and r % 2 == b]
    return [(r * cols + c, r * cols + c + cols) for r in range(rows - 1) for c in range(cols)
            if r % 2 == a and c % 2 == b]


def _zyz(rng):
    a, b, c = rng.uniform(0.0, 2 * math.pi, 3)
    z = [np.diag([np.exp(-0.5j * v), np.exp(0.5j * v)]) for v in (a, c)]
    y = np.array([[math.cos(b / 2), -math.sin(b / 2)], [math.sin(b / 2), math.cos(b / 2)]])
    return z[0] @ y @ z[1]


def _circuit(rows, cols, depth, seed, angles=False):
    """A random circuit of depth 1 + depth + 1: sqrt(X), sqrt(Y) and T drawn uniformly, or
    with `angles` a general rotation per qubit and cycle."""
    rng = np.random.default_rng([seed, rows, cols, depth])
    n = rows * cols
    gates = [Gate(0, q, -1, H, _MATS[H]) for q in range(n)]
    for t in range(depth):
        gates += [Gate(2 * t + 1, a, b, CZ, _CZ) for a, b in _pattern(rows, cols, t)]
        kinds = rng.integers(SQRT_X, T + 1, n)
        gates += [Gate(2 * t + 2, q, -1, U1, _zyz(rng)) if angles
                  else Gate(2 * t + 2, q, -1, int(kinds[q]), _MATS[int(kinds[q])]) for q in range(n)]
    gates += [Gate(2 * depth + 1, q, -1, H, _MATS[H]) for q in range(n)]
    return Grid(rows, cols, gates)


def _open_sites(rows, cols, n_open):
    """The last sites of a sweep along the shorter side (the library's own default)."""
    order = list(range(rows * cols)) if rows > cols else [r * cols + c for c in range(cols) for r in range(rows)]
    return order[len(order) - n_open:]


def _bits(n, count, rng):
    return rng.integers(0, 1 << n, count, dtype=np.int64)


def _plan(case, circuit):
    return qfx.Plan(qfx.Circuit(circuit), precision=case["precision"], family=case["family"],
                    open_sites=_open_sites(case["rows"], case["cols"], case["n_open"]),
                    max_intermediate_bytes=case["cap"])


# ------------------------------------------------------------------------------ the cases
def _amplitudes(rows, cols, depth, n_open, n_batch, in_flight, precision="fp32", family="line", cap=0,
                kind="amplitudes"):
    return dict(kind=kind, rows=rows, cols=cols, depth=depth, n_open=n_open, n_batch=n_batch,
                in_flight=in_flight, precision=precision, family=family, cap=cap)


def _step(precision, P, K, N, NL, Sd):
    return dict(kind="step", precision=precision, P=P, K=K, N=N, NL=NL, Sd=Sd)


def _permute(shape, perm):
    return dict(kind="permute", shape=",".join(map(str, shape)), perm=",".join(map(str, perm)))


def listed():
    return [
        # every amplitude of a 16-qubit circuit: a check of a small device; the launches and
        # the latency of tiny kernels count
        dict(name="amplitudes 4x4x16 all", **_amplitudes(4, 4, 16, 16, 1, 1)),
        # fast sampling of a 36-qubit circuit: 64 amplitudes and one sample per x1 batch
        dict(name="sample 6x6x24", **_amplitudes(6, 6, 24, 6, 37, 16, kind="sample")),
        # a training step: 128 amplitudes and the gradients of every gate
        dict(name="train 6x6x24", kind="train", rows=6, cols=6, depth=24, n_open=7, n_batch=1),
        # many small circuits at once
        dict(name="batch of small items", kind="batch", grids="4x4x16,4x5x16,5x5x24", items=24, n_open=4,
             n_batch=32, slots=304),
        # a deep 49-qubit circuit by the contraction tree, on the tensor cores
        dict(name="tree 7x7x28 bf16x3", **_amplitudes(7, 7, 28, 6, 1, 1, "bf16x3", "tree", 1 << 30)),
        # the dominant step of a depth-32 sweep (bond dimension 16), 1/32 of its columns
        dict(name="step fp32 chi16", **_step("fp32", 64, 256, 256, 256, 8192)),
        # a step of no round size, odd in every extent
        dict(name="step fp32 ragged", **_step("fp32", 7, 75, 99, 33, 4095)),
        # the same dominant step in the split precisions
        dict(name="step bf16x3 chi16", **_step("bf16x3", 64, 256, 256, 256, 8192)),
        dict(name="step tf32x3 chi16", **_step("tf32x3", 4096, 256, 256, 256, 128)),
        # the dominant step of an 11x11 grid's depth-24 sweep (bond dimension 8)
        dict(name="step bf16x3 chi8", **_step("bf16x3", 512, 64, 64, 64, 4096)),
        # a chunk of a tree's large contraction, at the quickest split
        dict(name="step bf16x2 chunk", **_step("bf16x2", 1, 1024, 1024, 1024, 32768)),
        # a reversal of seven axes: the transpose of a tree's operands
        dict(name="permute reversal", **_permute((16, 8, 32, 16, 8, 16, 16), (6, 5, 4, 3, 2, 1, 0))),
    ]


MOST_FLOPS = 3e11      # of a drawn case (the listed steps' 2.7e11, the tree's 1.6e12)
MOST_ELEMENTS = 1 << 27


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_step(rng):
    while True:
        prec = rng.choice(["fp32", "fp32", "bf16x3", "bf16x3", "tf32x3", "bf16x2"])
        if rng.random() < 0.5:     # a sweep's step: powers of two
            K, N, Sd = 1 << rng.randint(2, 10), 1 << rng.randint(2, 10), 1 << rng.randint(0, 16)
            NL = N >> rng.randint(0, 1)
        elif prec == "fp32":
            K, Sd = _log(rng, 2, 600), _log(rng, 1, 50000)
            NL = _log(rng, 2, 300)
            N = NL * rng.randint(1, 3)
        else:                      # what the tensor-core tiles take, of no round size
            K, N, Sd = 16 * _log(rng, 1, 40), 16 * _log(rng, 1, 8), _log(rng, 1, 50000)
            NL = N
        P = _log(rng, 1, 1 << 15)
        if P * Sd >= 128 and max(P * K * Sd, P * N * Sd) <= MOST_ELEMENTS and 8.0 * P * K * N * Sd <= MOST_FLOPS:
            return _step(prec, P, K, N, NL, Sd)


def _draw_permute(rng):
    rank = rng.randint(2, 7)
    goal = _log(rng, 1 << 12, MOST_ELEMENTS)
    while True:
        top = max(2, int(goal ** (1.0 / rank) * 3))
        shape = [1 << rng.randint(1, max(1, top.bit_length() - 1)) if rng.random() < 0.6 else rng.randint(2, top)
                 for _ in range(rank)]
        if goal / 4 <= math.prod(shape) <= goal:
            break
    perm = list(range(rank))
    while perm == sorted(perm):
        rng.shuffle(perm)
    return _permute(shape, perm)


def _draw_amplitudes(rng, kind):
    while True:
        rows, cols, depth = rng.randint(2, 6), rng.randint(3, 7), rng.randint(6, 28)
        n = rows * cols
        n_batch = _log(rng, 1, 40)
        case = _amplitudes(rows, cols, depth, rng.randint(0, min(n, 9)), n_batch, rng.randint(1, min(16, n_batch)),
                           rng.choice(["fp32", "fp32", "bf16x3", "tf32x3"]), kind=kind)
        if kind == "sample":
            case.update(precision="fp32", n_open=max(1, case["n_open"]))
        elif rng.random() < 0.4:
            case["family"] = "tree"
        if rng.random() < 0.2:
            case["cap"] = 1 << rng.randint(16, 24)
        try:
            plan = _plan(case, _circuit(rows, cols, depth, 0))
        except qfx.QfxError:       # no plan under this cap
            continue
        s = plan.stats
        work = s["n_slices"] * n_batch
        if work <= 512 and s["flops_per_item"] * work <= MOST_FLOPS and s["max_elements"] <= 1 << 25:
            return case


def draw(rng: random.Random):
    kind = rng.choice(["step"] * 8 + ["permute"] * 3 + ["amplitudes"] * 5 + ["sample", "train", "train", "batch"])
    if kind == "step":
        return _draw_step(rng)
    if kind == "permute":
        return _draw_permute(rng)
    if kind == "train":
        return dict(kind="train", rows=rng.randint(3, 6), cols=rng.randint(3, 6), depth=rng.randint(6, 24),
                    n_open=rng.randint(0, 8), n_batch=rng.randint(1, 3))
    if kind == "batch":
        grids = ["%dx%dx%d" % (rng.randint(3, 5), rng.randint(3, 5), rng.randint(8, 24)) for _ in range(rng.randint(1, 4))]
        return dict(kind="batch", grids=",".join(grids), items=rng.randint(len(grids), 30), n_open=rng.randint(0, 6),
                    n_batch=_log(rng, 1, 32), slots=rng.choice([16, 64, 304]))
    return _draw_amplitudes(rng, kind)


# ------------------------------------------------------------------------------ prepare, run
def _numbers(text):
    return [int(v) for v in text.split(",")]


def _randn(n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(n, dtype=torch.complex64, device="cuda", generator=g)


def _step_inputs(case, seed):
    return (_randn(case["K"] * case["N"], 2 * seed).view(case["K"], case["N"]),
            _randn(case["P"] * case["K"] * case["Sd"], 2 * seed + 1).view(case["P"], case["K"], case["Sd"]))


def _permute_input(case, seed):
    return _randn(math.prod(_numbers(case["shape"])), seed)


def _grid_input(case, seed):
    """The circuit and the x1 bitstrings (host) of a case on one grid."""
    rng = np.random.default_rng([seed, 1])
    return (_circuit(case["rows"], case["cols"], case["depth"], seed, case["kind"] == "train"),
            _bits(case["rows"] * case["cols"], case["n_batch"], rng), rng)


def _batch_inputs(case, seed):
    """(circuits, x1 bitstrings of every item): item i is of grid i mod the number of grids."""
    rng = np.random.default_rng([seed, 2])
    grids = [tuple(int(v) for v in g.split("x")) for g in case["grids"].split(",")]
    circuits = [_circuit(r, c, d, seed) for r, c, d in grids]
    return circuits, [_bits(grids[i % len(grids)][0] * grids[i % len(grids)][1], case["n_batch"], rng)
                      for i in range(case["items"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        S, B = _step_inputs(case, seed)
        need = qfx.qfx.step_scratch_bytes(case["K"], case["N"], case["precision"])
        return dict(case=case, S=S, B=B, out=torch.empty(case["P"] * case["N"] * case["Sd"], dtype=torch.complex64, device="cuda"),
                    scratch=torch.empty(need, dtype=torch.uint8, device="cuda") if need else None)
    if kind == "permute":
        x = _permute_input(case, seed)
        return dict(case=case, x=x, out=torch.empty_like(x), shape=_numbers(case["shape"]), perm=_numbers(case["perm"]))
    if kind == "batch":
        circuits, xs = _batch_inputs(case, seed)
        plans = [qfx.Plan(qfx.Circuit(c), open_sites=_open_sites(c.rows, c.cols, case["n_open"])) for c in circuits]
        items = [(plans[i % len(plans)], torch.from_numpy(x).cuda(), 0, None) for i, x in enumerate(xs)]
        return dict(case=case, batch=qfx.Batch(items, slots=case["slots"]))
    circuit, x1, rng = _grid_input(case, seed)
    state = dict(case=case, x1=torch.from_numpy(x1).cuda())
    if kind == "train":
        gates = np.array([g.mat.reshape(-1)[:4] for g in circuit.gates])
        return dict(state, template=circuit, gates=torch.from_numpy(gates).cuda().requires_grad_(True),
                    open_sites=_open_sites(case["rows"], case["cols"], case["n_open"]))
    plan = _plan(case, circuit)
    items = min(case["in_flight"], case["n_batch"] * plan.n_slices)
    state.update(plan=plan, workspace=torch.empty(plan.workspace_bytes(items), dtype=torch.uint8, device="cuda"))
    if kind == "sample":
        shape = (case["n_batch"], 1 << case["n_open"])
        state.update(mask=torch.from_numpy(_bits(case["n_open"], case["n_batch"], rng)).cuda(),
                     u=torch.from_numpy(rng.random(shape)).cuda())
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        return qfx.contract_step(state["S"], state["B"], case["P"], case["K"], case["N"], case["NL"], case["Sd"],
                                 precision=case["precision"], out=state["out"], scratch=state["scratch"])
    if kind == "permute":
        return qfx.permute(state["x"], state["shape"], state["perm"], out=state["out"])
    if kind == "batch":
        return state["batch"].run()
    if kind == "train":
        state["gates"].grad = None
        amps = qfx.circuit_amplitudes(state["gates"], state["template"], state["x1"], open_sites=state["open_sites"])
        amps.abs().square().sum().backward()
        return {"amps": amps.detach(), "grad": state["gates"].grad}
    if kind == "sample":
        x2, bits, amps = qfx.frugal_sample(state["plan"], state["x1"], state["u"], state["mask"],
                                           workspace=state["workspace"])
        return {"x2": x2, "bits": bits, "amps": amps}
    return qfx.amplitudes(state["plan"], state["x1"], workspace=state["workspace"])


# ------------------------------------------------------------------------------ work
def work(case):
    """Eq. 1's flops of the plan's contractions (8 per complex multiply-add; a gradient takes
    the forward sweep, the reverse sweep and the site gradients), and the bytes of the inputs
    (gates, bitstrings, operands) and outputs."""
    kind = case["kind"]
    if kind == "step":
        p, k, n, s = case["P"], case["K"], case["N"], case["Sd"]
        return {"bytes": 8.0 * (k * n + p * k * s + p * n * s), "flops": 8.0 * p * k * n * s}
    if kind == "permute":
        return {"bytes": 16.0 * math.prod(_numbers(case["shape"])), "flops": 0}
    if kind == "batch":
        circuits, _ = _batch_inputs(case, 0)
        each = [qfx.Plan(qfx.Circuit(c), open_sites=_open_sites(c.rows, c.cols, case["n_open"])).stats["flops_per_item"]
                for c in circuits]
        flops = sum(each[i % len(each)] for i in range(case["items"])) * case["n_batch"]
        return {"bytes": sum(64.0 * len(c.gates) for c in circuits)
                + case["items"] * case["n_batch"] * (8.0 + 16.0 * (1 << case["n_open"])), "flops": flops}
    circuit = _circuit(case["rows"], case["cols"], case["depth"], 0)
    gates, rows = 64.0 * len(circuit.gates), float(case["n_batch"] << case["n_open"])
    if kind == "train":
        plan = qfx.Plan(qfx.Circuit(circuit), open_sites=_open_sites(case["rows"], case["cols"], case["n_open"]))
        return {"bytes": 2 * gates + 8.0 * case["n_batch"] + 16.0 * rows,
                "flops": 3 * plan.stats["flops_per_item"] * case["n_batch"]}
    s = _plan(case, circuit).stats
    return {"bytes": gates + 8.0 * case["n_batch"] + 16.0 * rows + (24.0 * rows if kind == "sample" else 0),
            "flops": s["flops_per_item"] * s["n_slices"] * case["n_batch"]}


# ------------------------------------------------------------------------------ exact values
def _state_vector(circuit):
    """Amplitudes of all bitstrings, complex128: axis q of the result is qubit q."""
    n = circuit.rows * circuit.cols
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1
    for g in circuit.gates:
        m = torch.from_numpy(np.asarray(g.mat, dtype=np.complex128)).cuda()
        if g.q1 < 0:      # axis q has 2^(n-1-q) entries below it
            psi = torch.einsum("ab,xby->xay", m, psi.view(1 << g.q0, 2, -1)).reshape(-1)
        else:             # q0 < q1
            v = psi.view(1 << g.q0, 2, 1 << (g.q1 - g.q0 - 1), 2, -1)
            psi = (v * m.view(1, 2, 1, 2, 1)).reshape(-1)
    return psi.view([2] * n)


def _site_tensors(circuit, mats):
    """One tensor per qubit, axes [x] + one of extent 2 for every CZ on it, and their labels
    (gate index): CZ = sum over k of |k><k| on its first qubit and diag(D(k, .)) on the second."""
    n = circuit.rows * circuit.cols
    dev = mats.device
    site = [torch.tensor([1, 0], dtype=torch.complex128, device=dev) for _ in range(n)]
    legs = [[] for _ in range(n)]
    eye = torch.eye(2, dtype=torch.complex128, device=dev)
    for i, g in enumerate(circuit.gates):
        m = mats[i].view(2, 2)
        if g.q1 < 0:
            site[g.q0] = torch.tensordot(m, site[g.q0], dims=([1], [0]))
        else:
            for q, w in ((g.q0, eye), (g.q1, m.T)):     # w[b][k]
                site[q] = site[q].unsqueeze(-1) * w.view([2] + [1] * (site[q].dim() - 1) + [2])
                legs[q].append(i)
    return site, legs


def _pair_legs(circuit, site, legs):
    """Legs of one pair of neighbours merged into one axis; labels are the pairs, in order."""
    out = []
    for q, (t, ls) in enumerate(zip(site, legs)):
        pairs = {}
        for axis, i in enumerate(ls):
            g = circuit.gates[i]
            pairs.setdefault((g.q0, g.q1), []).append(axis + 1)
        t = t.permute([0] + [a for p in pairs for a in pairs[p]])
        out.append((t.reshape([2] + [1 << len(pairs[p]) for p in pairs]), [("x", q)] + list(pairs)))
    return out


def _order(shapes, tries=64):
    """A contraction order of labelled tensors [{label: extent}]: the pair that shares a label
    and whose result grows least over its operands, again and again; the one of least work of
    `tries` such runs, all but the first with the scores perturbed."""
    size = lambda t: math.prod(t.values())  # noqa: E731
    least, rng = None, random.Random(1)
    for attempt in range(tries):
        live, order, work = dict(enumerate(shapes)), [], 0
        noise = 0.0 if attempt == 0 else rng.choice([0.5, 1.0, 2.0])
        while len(live) > 1 and (least is None or work < least[0]):
            best = None
            for a in live:
                for b in live:
                    if a < b and (len(live) == 2 or any(k in live[b] for k in live[a])):
                        r = {k: v for t, u in ((live[a], live[b]), (live[b], live[a])) for k, v in t.items() if k not in u}
                        cost = math.log2(size(r)) - math.log2(max(size(live[a]), size(live[b]))) + noise * rng.random()
                        if best is None or cost < best[0]:
                            best = (cost, a, b, r)
            if best is None:      # parts that share nothing
                a, b = sorted(live)[:2]
                best = (0, a, b, {**live[a], **live[b]})
            _, a, b, r = best
            order.append((a, b))
            work += size({**live[a], **live[b]})
            del live[b]
            live[a] = r
        if len(live) == 1 and (least is None or work < least[0]):
            least = (work, order)
    return least[1]


def _network_order(tensors, open_sites):
    return _order([{k: s for k, s in zip(ls, t.shape) if k[0] != "x" or k[1] in open_sites} for t, ls in tensors])


def _network(tensors, order, x1, open_sites):
    """Amplitudes [2^n_open] of one x1 from merged site tensors, bit i of the index being the
    value of open_sites[i]."""
    live = {}
    for q, (t, labels) in enumerate(tensors):
        if q in open_sites:
            live[q] = (t, list(labels))
        else:
            live[q] = (t[(int(x1) >> q) & 1], list(labels[1:]))
    for a, b in order:
        (ta, la), (tb, lb) = live[a], live.pop(b)
        both = [k for k in la if k in lb]
        r = torch.tensordot(ta, tb, dims=([la.index(k) for k in both], [lb.index(k) for k in both]))
        live[a] = (r, [k for k in la if k not in both] + [k for k in lb if k not in both])
    t, labels = live[order[-1][0] if order else 0]
    return t.permute([labels.index(("x", q)) for q in reversed(open_sites)]).reshape(-1)


def _exact_amplitudes(circuit, x1, open_sites, cache=None):
    """[n_batch, 2^n_open] complex128."""
    n = circuit.rows * circuit.cols
    if n > 25:
        mats = torch.from_numpy(np.array([g.mat.reshape(-1)[:4] for g in circuit.gates])).cuda()
        tensors = _pair_legs(circuit, *_site_tensors(circuit, mats))
        order = _network_order(tensors, open_sites)
        return torch.stack([_network(tensors, order, x, open_sites) for x in x1])
    cache = {} if cache is None else cache
    if id(circuit) not in cache:
        cache[id(circuit)] = _state_vector(circuit)
    psi, rows = cache[id(circuit)], []
    for x in x1:
        row = psi[tuple(slice(None) if q in open_sites else (int(x) >> q) & 1 for q in range(n))]
        kept = sorted(open_sites)
        rows.append(row.permute([kept.index(q) for q in reversed(open_sites)]).reshape(-1))
    return torch.stack(rows)


def exact(case, seed):
    kind = case["kind"]
    if kind == "permute":
        x = _permute_input(case, seed).view(_numbers(case["shape"]))
        return x.permute(_numbers(case["perm"])).contiguous().view(-1)
    if kind == "step":
        S, B = (v.to(torch.complex128) for v in _step_inputs(case, seed))
        p, k, n, nl, s = (case[v] for v in ("P", "K", "N", "NL", "Sd"))
        out = torch.empty((n // nl, p, nl, s), dtype=torch.complex128, device="cuda")
        for i in range(p):
            out[:, i] = (S.T @ B[i]).view(n // nl, nl, s)
        return out.view(-1)
    if kind == "batch":
        circuits, xs = _batch_inputs(case, seed)
        cache = {}
        return [_exact_amplitudes(circuits[i % len(circuits)], x,
                                  _open_sites(circuits[i % len(circuits)].rows, circuits[i % len(circuits)].cols, case["n_open"]), cache)
                for i, x in enumerate(xs)]
    circuit, x1, _ = _grid_input(case, seed)
    sites = _open_sites(case["rows"], case["cols"], case["n_open"])
    if kind == "train":
        gates = torch.from_numpy(np.array([g.mat.reshape(-1)[:4] for g in circuit.gates])).cuda().requires_grad_(True)
        tensors = _pair_legs(circuit, *_site_tensors(circuit, gates))
        order = _network_order(tensors, sites)
        amps = torch.stack([_network(tensors, order, x, sites) for x in x1])
        amps.abs().square().sum().backward()
        return {"amps": amps.detach(), "grad": gates.grad}
    amps = _exact_amplitudes(circuit, x1, sites)
    return {"x2": None, "bits": None, "amps": amps} if kind == "sample" else amps
