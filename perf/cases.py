"""The work that users of this framework have it do, as cases to be timed.

Each case is one call (or one training step) through the public entry points
of ``paper_2602_11092_gb300``: a plan's forward pass, a ``QuantumLayer`` step,
a batch of uneven circuits, a Gram matrix, a batch of encoded states, shots,
the surrogate network.  Sizes come from this repository's workloads, tests and
benchmark.

``exact`` restates every case in 64 bits with plain torch: the Clements mesh
as row rotations, the photon-by-photon recursion as gathers over enumerated
Fock states with torch's own autograd for gradients, permanents by Glynn's
formula, a dense network.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2602_11092_gb300 as package

DEV = "cuda"


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # one call on the smallest circuit: nothing but launch and host latency
        {"name": "tiny_forward", "kind": "forward", "m": 6, "n": 3, "batch": 1, "detect": "pnr", "output": "probs"},
        # one large circuit simulated alone, all amplitudes wanted
        {"name": "single16_amps", "kind": "forward", "m": 16, "n": 8, "batch": 1, "detect": "pnr", "output": "amps"},
        # a layer's inference over a large batch: meshes, then every distribution
        {"name": "layer12_infer", "kind": "mesh_forward", "m": 12, "n": 6, "batch": 4096, "detect": "pnr"},
        # evaluation of a trained layer with click detectors, the module called without gradients, a ragged batch
        {"name": "threshold16_eval", "kind": "eval", "m": 16, "n": 6, "batch": 100, "detect": "threshold"},
        # an ordinary training step, a ragged batch: a loss that is not linear hands back a gradient row per instance
        {"name": "layer12_step", "kind": "step", "m": 12, "n": 6, "batch": 1000, "detect": "pnr", "space": "fock",
         "measure": "probs", "renormalise": False, "shared": False, "budget": 0},
        # the headline training step: a linear loss (one gradient row for the batch), activations checkpointed
        {"name": "train16_step", "kind": "step", "m": 16, "n": 8, "batch": 256, "detect": "pnr", "space": "fock",
         "measure": "probs", "renormalise": False, "shared": True, "budget": 1_950_000},
        # a layer on collision-free outputs, conditioned on them, that hands mode expectations to what follows
        {"name": "unbunched16_step", "kind": "step", "m": 16, "n": 6, "batch": 512, "detect": "pnr",
         "space": "unbunched", "measure": "expectations", "renormalise": True, "shared": False, "budget": 0},
        # circuits of many shapes in one persistent launch
        {"name": "uneven1024", "kind": "uneven", "count": 1024, "m_lo": 8, "m_hi": 20, "n_hi": 10, "shapes": 1003},
        # Gram matrix of a training set for a kernel method
        {"name": "gram1024", "kind": "gram", "m": 12, "n": 6, "points": 1024, "others": 0},
        # amplitude-encoded states through one unitary
        {"name": "encoded10", "kind": "encoded", "m": 10, "n": 5, "batch": 4096, "output": "probs"},
        # finite shots from simulated distributions, as a processor returns them
        {"name": "shots12", "kind": "shots", "m": 12, "n": 6, "batch": 256, "shots": 1000, "counts": True},
        # the learned surrogate of the 12-mode layer over a batch
        {"name": "surrogate12", "kind": "surrogate", "phases": 144, "hidden": 2048, "layers": 4, "outputs": 12376,
         "batch": 16384},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _states_upto(m, n, space="fock"):
    dim = _dim if space == "fock" else (lambda a, b: math.comb(a, b))
    return sum(dim(m, k) for k in range(1, n + 1))


# amplitudes of all layers of a drawn batch: below the listed training step's
_DRAW_STATES = 9.0e7


def draw(rng):
    kind = rng.choice(["forward", "mesh_forward", "eval", "step", "step", "step", "uneven", "gram", "encoded", "shots",
                       "surrogate"])
    if kind in ("forward", "mesh_forward", "eval", "step"):
        m = rng.randint(4, 18)
        n = rng.randint(2, max(2, min(8, m // 2 + 1)))
        space = "fock"
        if kind == "step" and rng.random() < 0.35:
            space = "unbunched"
        detect = "threshold" if space == "fock" and rng.random() < 0.3 else "pnr"
        most = max(1, int(_DRAW_STATES / _states_upto(m, n, space)))
        case = {"kind": kind, "m": m, "n": n, "batch": _log_int(rng, 1, min(most, 8192)), "detect": detect}
        if kind == "forward":
            case["output"] = "amps" if detect == "pnr" and rng.random() < 0.4 else "probs"
        if kind == "step":
            case["batch"] = min(case["batch"], 2048)
            case["space"] = space
            case["measure"] = "expectations" if rng.random() < 0.4 else "probs"
            case["renormalise"] = space == "unbunched" and rng.random() < 0.5
            case["shared"] = case["measure"] == "probs" and not case["renormalise"] and rng.random() < 0.3
            case["budget"] = 0
        return case
    if kind == "uneven":
        lo = rng.randint(6, 12)
        return {"kind": kind, "count": _log_int(rng, 16, 1000), "m_lo": lo, "m_hi": rng.randint(lo + 2, 17),
                "n_hi": rng.randint(4, 8), "shapes": rng.randint(1, 10 ** 6)}
    if kind == "gram":
        m = rng.randint(6, 16)
        return {"kind": kind, "m": m, "n": rng.randint(2, min(7, m // 2)), "points": _log_int(rng, 30, 1100),
                "others": rng.choice([0, 0, rng.randint(20, 700)])}
    if kind == "encoded":
        m, n = rng.choice([(6, 3), (7, 3), (8, 3), (8, 4), (9, 4), (10, 4), (11, 4), (10, 5)])
        return {"kind": kind, "m": m, "n": n, "batch": _log_int(rng, 16, 4000),
                "output": rng.choice(["probs", "amps"])}
    if kind == "shots":
        m = rng.randint(6, 16)
        n = rng.randint(2, min(7, m // 2))
        most = max(1, int(8.0e6 / _dim(m, n)))
        return {"kind": kind, "m": m, "n": n, "batch": _log_int(rng, 1, min(most, 4096)),
                "shots": _log_int(rng, 10, 4000), "counts": rng.random() < 0.5}
    return {"kind": "surrogate", "phases": 4 * rng.randint(9, 36), "hidden": 256 * rng.randint(1, 8),
            "layers": rng.randint(2, 4), "outputs": 8 * rng.randint(40, 1547), "batch": 8 * _log_int(rng, 16, 1600)}


# ------------------------------------------------------------- what a user has

def _dim(m, n):
    return math.comb(m + n - 1, n)


def _input_state(m, n):
    """n photons over the even modes first, then the odd ones (bunching beyond m)."""
    order = list(range(0, m, 2)) + list(range(1, m, 2))
    s = [0] * m
    for i in range(n):
        s[order[i % m]] += 1
    return s


def _haar(m, count, gen):
    z = torch.complex(torch.randn(count, m, m, generator=gen, dtype=torch.float64),
                      torch.randn(count, m, m, generator=gen, dtype=torch.float64))
    q, r = torch.linalg.qr(z)
    d = torch.diagonal(r, dim1=-2, dim2=-1)
    return (q * (d / d.abs()).unsqueeze(-2)).to(torch.complex64).contiguous()


def _phases(m, batch, gen):
    """Trainable phases U(0, 2 pi), encoding weights U(0, pi), features N(0, 1)."""
    theta = torch.rand(m * (m - 1), generator=gen) * (2 * math.pi)
    w = torch.rand(m, generator=gen) * math.pi
    x = torch.randn(batch, m, generator=gen)
    return theta.to(DEV), w.to(DEV), x.to(DEV)


def _n_outputs(case):
    m, n = case["m"], case["n"]
    if case.get("detect") == "threshold":
        return sum(math.comb(m, k) for k in range(1, min(m, n) + 1))
    return math.comb(m, n) if case.get("space") == "unbunched" else _dim(m, n)


def _uneven_shapes(case):
    rng = np.random.default_rng(case["shapes"])
    shapes = []
    for _ in range(case["count"]):
        m = int(rng.integers(case["m_lo"], case["m_hi"] + 1))
        shapes.append((m, int(rng.integers(2, min(case["n_hi"], m // 2) + 1)), m >= 16))
    return shapes


def _uneven_unitaries(case, gen):
    """One Haar unitary per instance, instance by instance in the packed order."""
    shapes = _uneven_shapes(case)
    Us = [None] * len(shapes)
    for m in sorted({s[0] for s in shapes}):
        at = [i for i, s in enumerate(shapes) if s[0] == m]
        for i, u in zip(at, _haar(m, len(at), gen)):
            Us[i] = u
    return shapes, Us


def _inputs(case, seed):
    """The case's tensors, made from the seed alone."""
    gen = torch.Generator().manual_seed(int(seed))
    kind = case["kind"]
    if kind == "forward":
        return {"U": _haar(case["m"], case["batch"], gen).to(DEV)}
    if kind in ("mesh_forward", "eval", "step"):
        theta, w, x = _phases(case["m"], case["batch"], gen)
        got = {"theta": theta, "w": w, "x": x}
        if kind == "step":
            width = case["m"] if case["measure"] == "expectations" else _n_outputs(case)
            rows = 1 if case["shared"] else case["batch"]
            on_card = torch.Generator(device=DEV).manual_seed(int(seed))
            got["grad"] = torch.randn(rows, width, generator=on_card, device=DEV)
        return got
    if kind == "uneven":
        shapes, Us = _uneven_unitaries(case, gen)
        return {"shapes": shapes, "U": torch.cat([u.reshape(-1) for u in Us]).to(DEV)}
    if kind == "gram":
        theta, w, x = _phases(case["m"], case["points"], gen)
        other = torch.randn(case["others"], case["m"], generator=gen).to(DEV) if case["others"] else None
        return {"theta": theta, "w": w, "x": x, "other": other}
    if kind == "encoded":
        K = _dim(case["m"], case["n"])
        on_card = torch.Generator(device=DEV).manual_seed(int(seed))
        X = torch.complex(torch.randn(case["batch"], K, generator=on_card, device=DEV),
                          torch.randn(case["batch"], K, generator=on_card, device=DEV))
        X = X / torch.linalg.vector_norm(X, dim=1, keepdim=True)
        return {"U": _haar(case["m"], 1, gen)[0].to(DEV), "X": X}
    if kind == "shots":
        K = _dim(case["m"], case["n"])
        on_card = torch.Generator(device=DEV).manual_seed(int(seed))
        p = torch.empty(case["batch"], K, device=DEV).exponential_(generator=on_card)
        p = p * torch.empty(case["batch"], K, device=DEV).exponential_(generator=on_card)
        p = p / p.sum(dim=1, keepdim=True)
        u = torch.rand(case["batch"], case["shots"], generator=on_card, device=DEV)
        return {"p": p, "u": u}
    # surrogate: a network of the case's shape, He-uniform weights, small biases
    on_card = torch.Generator(device=DEV).manual_seed(int(seed))
    layers = []
    fan_in = 2 * case["phases"]
    for layer in range(case["layers"] + 1):
        fan_out = case["outputs"] if layer == case["layers"] else case["hidden"]
        lim = math.sqrt(6.0 / fan_in)
        layers.append(((torch.rand(fan_out, fan_in, generator=on_card, device=DEV) * 2 - 1) * lim,
                       (torch.rand(fan_out, generator=on_card, device=DEV) * 2 - 1) * 0.1))
        fan_in = fan_out
    phases = torch.randn(case["batch"], case["phases"], generator=on_card, device=DEV) * 2.0
    return {"layers": layers, "phases": phases}


def _layer(case, data):
    from paper_2602_11092_gb300 import binding as B
    from paper_2602_11092_gb300.functions import QuantumLayer
    return QuantumLayer(case["m"], _input_state(case["m"], case["n"]),
                        B.THRESHOLD if case["detect"] == "threshold" else B.PNR,
                        mem_budget_bytes=case.get("budget", 0), theta=data["theta"], w=data["w"], device=DEV,
                        space=B.UNBUNCHED if case.get("space") == "unbunched" else B.FOCK,
                        renormalise=case.get("renormalise", False), measurement=case.get("measure"))


def prepare(case, seed):
    B = package.load()
    data = _inputs(case, seed)
    kind = case["kind"]
    state = {"case": case, "B": B}
    if kind in ("forward", "mesh_forward"):
        state["plan"] = B.Plan(case["m"], _input_state(case["m"], case["n"]),
                               B.THRESHOLD if case["detect"] == "threshold" else B.PNR)
        state.update(data)
        if kind == "mesh_forward":
            state["phases"] = (data["x"] * data["w"]).contiguous()
    elif kind == "eval":
        state["layer"] = _layer(case, data)
        state["x"] = data["x"]
    elif kind == "step":
        state["layer"] = _layer(case, data)
        state["x"] = data["x"].requires_grad_(True)
        state["grad"] = data["grad"].expand(case["batch"], -1)
    elif kind == "uneven":
        shapes = data["shapes"]
        plan = B.BatchedPlan([s[0] for s in shapes], [s[1] for s in shapes],
                             [_input_state(s[0], s[1]) for s in shapes],
                             [B.THRESHOLD if s[2] else B.PNR for s in shapes])
        state.update(plan=plan, U=data["U"], out=torch.empty(plan.out_offsets[-1], device=DEV),
                     workspace=torch.empty(plan.workspace_bytes, dtype=torch.uint8, device=DEV))
    elif kind == "gram":
        from paper_2602_11092_gb300.functions import FidelityKernel
        state["kernel"] = FidelityKernel(case["m"], _input_state(case["m"], case["n"]), theta=data["theta"],
                                         w=data["w"], device=DEV)
        state.update(x=data["x"], other=data["other"])
    elif kind == "encoded":
        plan = B.Plan(case["m"], _input_state(case["m"], case["n"]))
        state.update(plan=plan, workspace=torch.empty(plan.encoded_workspace_bytes(), dtype=torch.uint8, device=DEV),
                     **data)
    elif kind == "shots":
        state.update(plan=B.Plan(case["m"], _input_state(case["m"], case["n"])), **data)
    else:
        from paper_2602_11092_gb300.surrogate import Surrogate
        model = Surrogate(n_phases=case["phases"], hidden=case["hidden"], n_hidden_layers=case["layers"],
                          n_outputs=case["outputs"], max_batch=case["batch"])
        for i, (weight, bias) in enumerate(data["layers"]):
            model.set_param(i, weight.cpu().numpy(), bias.cpu().numpy())
        state.update(model=model, phases=data["phases"])
    return state


def run(state):
    case, B = state["case"], state["B"]
    kind = case["kind"]
    if kind == "forward":
        return state["plan"].forward(state["U"], B.AMPS if case["output"] == "amps" else B.PROBS)
    if kind == "mesh_forward":
        U = B.mesh_unitary(case["m"], state["theta"], state["phases"], case["batch"])
        return state["plan"].forward(U)
    if kind == "eval":
        with torch.no_grad():
            return state["layer"](state["x"])
    if kind == "step":
        layer, x = state["layer"], state["x"]
        y = layer(x)
        dtheta, dx = torch.autograd.grad(y, (layer.theta, x), state["grad"])
        return [y, dtheta, dx]
    if kind == "uneven":
        return state["plan"].forward(state["U"], state["out"], state["workspace"])
    if kind == "gram":
        return state["kernel"](state["x"], state["other"])
    if kind == "encoded":
        return state["plan"].encoded_forward(state["U"], state["X"], B.AMPS if case["output"] == "amps" else B.PROBS,
                                             workspace=state["workspace"])
    if kind == "shots":
        got = state["plan"].sample(state["p"], state["u"], counts=case["counts"])
        return list(got) if case["counts"] else got
    return state["model"].forward(state["phases"])


# ---------------------------------------------------------- what a pass needs

def _recursion_flops(m, n, space="fock"):
    """A complex multiply-add (8) for every edge of the photon-by-photon recursion of one instance."""
    if space == "unbunched":
        return 8.0 * sum(k * math.comb(m, k) for k in range(1, n + 1))
    return 8.0 * m * sum(_dim(m, k) for k in range(n))


def _mesh_flops(m):
    """One column step: 4 complex multiply-adds on each of m columns, m (m - 1) / 2 rotations."""
    return 32.0 * m * (m * (m - 1) / 2)


def work(case):
    kind = case["kind"]
    if kind in ("forward", "mesh_forward", "eval", "step"):
        m, n, b = case["m"], case["n"], case["batch"]
        size = 8 if case.get("output") == "amps" else 4
        width = m if case.get("measure") == "expectations" else _n_outputs(case)
        flops = b * _recursion_flops(m, n, case.get("space", "fock"))
        if kind == "forward":
            return {"bytes": b * (8.0 * m * m + size * width), "flops": flops}
        P = m * (m - 1)
        data = 4.0 * (P + m + b * m)
        if kind != "step":
            return {"bytes": data + b * 4.0 * width, "flops": flops + b * _mesh_flops(m)}
        rows = 1 if case["shared"] else b
        return {"bytes": data + 4.0 * (b * width + rows * width + P + b * m),
                "flops": 3 * (flops + b * _mesh_flops(m))}
    if kind == "uneven":
        total, flops = 0.0, 0.0
        for m, n, threshold in _uneven_shapes(case):
            K = sum(math.comb(m, k) for k in range(1, n + 1)) if threshold else _dim(m, n)
            total += 8.0 * m * m + 4.0 * K
            flops += _recursion_flops(m, n)
        return {"bytes": total, "flops": flops}
    if kind == "gram":
        m, n, a = case["m"], case["n"], case["points"]
        # a matrix of a set against itself is symmetric
        c = case["others"]
        pairs = a * c if c else a * (a + 1) / 2
        per = 8.0 * m * n * n + 8.0 * n * 2 ** (n - 1)
        return {"bytes": 4.0 * (m * (a + c) + a * (c or a)), "flops": pairs * per + (a + c) * _mesh_flops(m)}
    if kind == "encoded":
        m, n, b = case["m"], case["n"], case["batch"]
        K = _dim(m, n)
        size = 8 if case["output"] == "amps" else 4
        return {"bytes": 8.0 * m * m + b * K * (8.0 + size), "flops": 8.0 * b * K * K}
    if kind == "shots":
        K, b, s = _dim(case["m"], case["n"]), case["batch"], case["shots"]
        return {"bytes": 4.0 * b * (K + 2 * s + (K if case["counts"] else 0)), "flops": float(b * K)}
    f, h, layers, K, b = 2 * case["phases"], case["hidden"], case["layers"], case["outputs"], case["batch"]
    weights = f * h + (layers - 1) * h * h + h * K
    return {"bytes": 4.0 * b * (case["phases"] + K) + 2.0 * weights, "flops": 2.0 * b * weights}


# ------------------------------------------------- the same numbers in 64 bits

def _fock_states(m, k, cache):
    """uint8 [F, m]: compositions of k photons over m modes, descending lexicographic order."""
    if (m, k) not in cache:
        if m == 1:
            cache[m, k] = torch.full((1, 1), k, dtype=torch.uint8, device=DEV)
        else:
            parts = []
            for first in range(k, -1, -1):
                rest = _fock_states(m - 1, k - first, cache)
                head = torch.full((rest.shape[0], 1), first, dtype=torch.uint8, device=DEV)
                parts.append(torch.cat([head, rest], dim=1))
            cache[m, k] = torch.cat(parts)
    return cache[m, k]


def _free_states(m, k):
    """uint8 [C(m, k), m]: collision-free states, descending lexicographic order, and their codes."""
    codes = torch.arange(1 << m, device=DEV)
    count = torch.zeros_like(codes)
    for j in range(m):
        count += (codes >> j) & 1
    codes = codes[count == k].flip(0)
    return torch.stack([(codes >> (m - 1 - j)) & 1 for j in range(m)], dim=1).to(torch.uint8), codes


def _fock_parents(states, m, k):
    """For each mode j: index in layer k - 1 of every state less one photon in j (F_{k-1} where it has none)."""
    after = torch.zeros(states.shape[0], dtype=torch.int64, device=DEV)  # photons after mode b
    left = [None] * m
    for b in range(m - 1, -1, -1):
        left[b] = after.clone()
        after += states[:, b].long()
    tables = [torch.tensor([math.comb(r + m - 2 - b, m - 1 - b) if r + m - 2 - b >= 0 else 0
                            for r in range(-1, k + 1)], device=DEV) for b in range(m - 1)]
    whole = torch.zeros_like(after)
    for b in range(m - 1):
        whole += tables[b][left[b] + 1]
    lowered = torch.zeros_like(after)  # modes before j: one photon fewer after them
    for j in range(m):
        yield torch.where(states[:, j] > 0, whole + lowered, _dim(m, k - 1))
        if j < m - 1:
            lowered += tables[j][left[j]] - tables[j][left[j] + 1]


def _free_parents(states, codes, m, k):
    before = _free_states(m, k - 1)[1].flip(0)
    for j in range(m):
        at = torch.searchsorted(before, codes - (1 << (m - 1 - j))).clamp(max=before.numel() - 1)
        yield torch.where(states[:, j] > 0, before.numel() - 1 - at, before.numel())


def _amplitudes(U, s, space, cache):
    """a_n [F_n, B] of unitaries U [B, m, m] for input s, and the states [F_n, m]."""
    m = len(s)
    cols = [c for c in range(m) for _ in range(s[c])]
    a = torch.ones(1, U.shape[0], dtype=torch.complex128, device=DEV)
    for k, c in enumerate(cols, 1):
        if space == "unbunched":
            states, codes = _free_states(m, k)
            parents = _free_parents(states, codes, m, k)
        else:
            states = _fock_states(m, k, cache)
            parents = _fock_parents(states, m, k)
        rows = torch.cat([a, torch.zeros(1, a.shape[1], dtype=a.dtype, device=DEV)])
        total = None
        for j, at in enumerate(parents):
            term = rows.index_select(0, at) * U[:, j, c]
            total = term if total is None else total + term
        a = total
    return a, states


def _weights(states, s):
    f = torch.ones(states.shape[0], dtype=torch.float64, device=DEV)
    table = torch.tensor([math.factorial(q) for q in range(sum(s) + 1)], dtype=torch.float64, device=DEV)
    for j in range(states.shape[1]):
        f = f * table[states[:, j].long()]
    return f / math.prod(math.factorial(q) for q in s)


def _patterns(states, n):
    """Index of every state's set of occupied modes: by size, then colex rank."""
    m = states.shape[1]
    size = torch.zeros(states.shape[0], dtype=torch.int64, device=DEV)
    rank = torch.zeros_like(size)
    choose = torch.tensor([[math.comb(q, i) for i in range(m + 2)] for q in range(m)], device=DEV)
    for q in range(m):
        on = (states[:, q] > 0).long()
        size += on
        rank += on * choose[q][size]
    starts = [0, 0]
    for i in range(1, min(m, n) + 1):
        starts.append(starts[-1] + math.comb(m, i))
    return torch.tensor(starts, device=DEV)[size] + rank, starts[-1]


def _distribution(U, s, detect, space, cache):
    """[B, K] probabilities, and the occupations [K, m] of the outcomes."""
    a, states = _amplitudes(U, s, space, cache)
    p = (a.real.square() + a.imag.square()) * _weights(states, s)[:, None]
    occ = states.double()
    if detect == "threshold":
        at, count = _patterns(states, sum(s))
        p = torch.zeros(count, p.shape[1], dtype=p.dtype, device=DEV).index_add(0, at, p)
        occ = torch.zeros(count, len(s), dtype=torch.float64, device=DEV).index_copy(0, at, (occ > 0).double())
    return p.T, occ


def _mesh(m, theta, phi):
    """[B, m, m] from 64-bit phases: m columns of rotations, the data screen in the middle."""
    X = torch.eye(m, dtype=torch.complex128, device=DEV).expand(phi.shape[0], m, m)
    at = 0
    for c in range(m + 1):
        if c == m // 2:
            X = X * torch.exp(1j * phi)[:, :, None]
        rows = torch.arange(c % 2, m - 1, 2, device=DEV)
        if c == m or not len(rows):
            continue
        t = theta[at:at + 2 * len(rows)].reshape(-1, 2)
        at += 2 * len(rows)
        half, e = t[:, 0] / 2, torch.exp(1j * t[:, 1])
        g = 1j * torch.exp(1j * half)
        sin, cos = (g * torch.sin(half))[:, None], (g * torch.cos(half))[:, None]
        e = e[:, None]
        top, low = X[:, rows], X[:, rows + 1]
        X = X.index_copy(1, rows, sin * e * top + cos * low).index_copy(1, rows + 1, cos * e * top - sin * low)
    return X


def _exact_step(case, data):
    m, s = case["m"], _input_state(case["m"], case["n"])
    theta = data["theta"].double().requires_grad_(True)
    w = data["w"].double()
    cache = {}
    # autograd keeps every gathered row: a slice of the batch at a time
    per = max(1, min(case["batch"], int(2.0e7 / _n_outputs({**case, "detect": "pnr"}))))
    ys, dxs, dtheta = [], [], torch.zeros_like(theta)
    for b in range(0, case["batch"], per):
        x = data["x"][b:b + per].detach().double().requires_grad_(True)
        y, occ = _distribution(_mesh(m, theta, x * w), s, case["detect"], case["space"], cache)
        if case["renormalise"]:
            y = y / y.sum(dim=1, keepdim=True)
        if case["measure"] == "expectations":
            y = y @ occ
        g = data["grad"].double()
        g = g.expand(y.shape) if case["shared"] else g[b:b + per]
        dt, dx = torch.autograd.grad(y, (theta, x), g)
        dtheta += dt
        ys.append(y.detach())
        dxs.append(dx)
    return [torch.cat(ys), dtheta.detach(), torch.cat(dxs)]


def _exact_batches(case, s, U_of, amps=False):
    """Forward outputs, a slice of the batch at a time."""
    cache, got = {}, []
    per = max(1, int(1.0e8 / _dim(case["m"], case["n"])))
    for b in range(0, case["batch"], per):
        U = U_of(b, min(case["batch"], b + per))
        if amps:
            a, states = _amplitudes(U, s, "fock", cache)
            got.append((a * _weights(states, s).sqrt()[:, None]).T.contiguous())
        else:
            got.append(_distribution(U, s, case["detect"], "fock", cache)[0].contiguous())
    return torch.cat(got)


def _exact_uneven(data):
    shapes, U = data["shapes"], data["U"].to(torch.complex128)
    starts, offsets, at, off = [], [], 0, 0
    for m, n, threshold in shapes:
        starts.append(at)
        offsets.append(off)
        at += m * m
        off += sum(math.comb(m, k) for k in range(1, n + 1)) if threshold else _dim(m, n)
    out = torch.empty(off, dtype=torch.float64, device=DEV)
    for m in sorted({s[0] for s in shapes}):
        cache = {}
        for n in sorted({s[1] for s in shapes if s[0] == m}):
            some = [i for i, s in enumerate(shapes) if s[:2] == (m, n)]
            per = max(1, int(6.0e7 / _dim(m, n)))
            for b in range(0, len(some), per):
                part = some[b:b + per]
                V = torch.stack([U[starts[i]:starts[i] + m * m].reshape(m, m) for i in part])
                p, _ = _distribution(V, _input_state(m, n), "threshold" if m >= 16 else "pnr", "fock", cache)
                for i, row in zip(part, p):
                    out[offsets[i]:offsets[i] + row.numel()] = row
    return out


def _exact_gram(case, data):
    m, n = case["m"], case["n"]
    s = _input_state(m, n)
    cols = torch.tensor([c for c in range(m) for _ in range(s[c])], device=DEV)
    theta, w = data["theta"].double(), data["w"].double()
    A = _mesh(m, theta, data["x"].double() * w)[:, :, cols]
    C = A if data["other"] is None else _mesh(m, theta, data["other"].double() * w)[:, :, cols]
    rows = []
    for a in A.split(64):
        W = torch.einsum("ikr,jkc->ijrc", a.conj(), C)
        per = torch.zeros(W.shape[:2], dtype=torch.complex128, device=DEV)
        for code in range(2 ** (n - 1)):
            signs = [1] + [-1 if (code >> q) & 1 else 1 for q in range(n - 1)]
            delta = torch.tensor(signs, dtype=torch.complex128, device=DEV)
            per = per + math.prod(signs) * torch.einsum("r,ijrc->ijc", delta, W).prod(dim=2)
        per = per / 2 ** (n - 1) / math.prod(math.factorial(q) for q in s)
        rows.append(per.abs().square())
    return torch.cat(rows)


def _exact_encoded(case, data):
    """The transfer matrix A_k[t, s] of every input s, layer by layer, then one product."""
    m, n = case["m"], case["n"]
    U = data["U"].to(torch.complex128)
    cache = {}
    A = torch.ones(1, 1, dtype=torch.complex128, device=DEV)
    for k in range(1, n + 1):
        states = _fock_states(m, k, cache)
        parents = list(_fock_parents(states, m, k))
        modes = torch.arange(m, device=DEV)
        last = torch.where(states > 0, modes, -1).max(dim=1).values  # highest occupied mode of the input
        source = torch.stack(parents)[last, torch.arange(states.shape[0], device=DEV)]
        rows = torch.cat([A, torch.zeros(1, A.shape[1], dtype=A.dtype, device=DEV)]).index_select(1, source)
        A = sum(rows.index_select(0, at) * U[j, last] for j, at in enumerate(parents))
    root = _weights(states, [0] * m + [n]).mul(math.factorial(n)).sqrt()  # sqrt(prod t!)
    psi = (data["X"].to(torch.complex128) / root) @ A.T * root
    return psi if case["output"] == "amps" else psi.abs().square()


def _exact_surrogate(case, data):
    got = []
    layers = [(a.double(), b.double()) for a, b in data["layers"]]
    for phases in data["phases"].split(4096):
        h = phases.double()
        h = torch.cat([torch.sin(h), torch.cos(h)], dim=1)
        for i, (a, b) in enumerate(layers):
            h = h @ a.T + b
            if i < len(layers) - 1:
                h = torch.nn.functional.gelu(h, approximate="tanh")
        got.append(torch.softmax(h, dim=1))
    return torch.cat(got)


def exact(case, seed):
    data = _inputs(case, seed)
    kind = case["kind"]
    if kind == "step":
        return _exact_step(case, data)
    with torch.no_grad():
        if kind == "forward":
            return _exact_batches(case, _input_state(case["m"], case["n"]),
                                  lambda b, e: data["U"][b:e].to(torch.complex128), case["output"] == "amps")
        if kind in ("mesh_forward", "eval"):
            theta, w = data["theta"].double(), data["w"].double()
            # the inference call is handed x * w as formed in 32 bits, the module forms it itself
            phi = (data["x"] * data["w"]).double() if kind == "mesh_forward" else data["x"].double() * w
            return _exact_batches(case, _input_state(case["m"], case["n"]),
                                  lambda b, e: _mesh(case["m"], theta, phi[b:e]))
        if kind == "uneven":
            return _exact_uneven(data)
        if kind == "gram":
            return _exact_gram(case, data)
        if kind == "encoded":
            return _exact_encoded(case, data)
        if kind == "shots":
            return None  # outcome indices and counts: whole numbers
        return _exact_surrogate(case, data)
