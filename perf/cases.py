"""The work that users of this package have it do, as measurable cases.

A case is a dict of plain values; `prepare` builds what a program holds before
the call (states, packed circuits and Hamiltonians, batch handles, angles),
`run` makes one pass through the package's public calls, `work` says what the
pass cannot do without and `exact` computes its outputs in 64 bits with plain
torch.

Results that a complex64 state determines (energies, gradients) are returned
as float32, the precision they carry; complex128 results stay 64-bit.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2202_07017_gb300 import Batch, State, energy, pack_circuit, pack_pauli


# ---- the cases ---------------------------------------------------------------------------
def listed():
    return [
        # a small circuit, one kernel per gate, double precision: launches and latency decide
        {"name": "layered_n12_c128", "kind": "layered", "n": 12, "depth": 20, "dtype": "c128", "fuse": 0},
        # the quantum Fourier transform gate by gate on a state far above the caches
        {"name": "qft_n30_c64", "kind": "qft", "n": 30, "dtype": "c64", "fuse": 0},
        # the same in double precision, an odd qubit count
        {"name": "qft_n27_c128", "kind": "qft", "n": 27, "dtype": "c128", "fuse": 0},
        # a deep random circuit with gate fusion: the large simulations
        {"name": "layered_n28_c64_fused", "kind": "layered", "n": 28, "depth": 30, "dtype": "c64", "fuse": 4},
        # one variational training step (energy and gradient through autograd) of the
        # hardware-efficient ansatz
        {"name": "hea_grad_n20", "kind": "hea_grad", "n": 20, "depth": 10, "dtype": "c64", "fuse": 4},
        # gradient of a deep circuit on a large state with forward checkpoints
        {"name": "layered_grad_n26", "kind": "layered_grad", "n": 26, "depth": 12, "every": 4,
         "dtype": "c64", "fuse": 4},
        # many variational solves at once: parameter sets of one ansatz plus a mixed
        # population of sizes and depths (every gate and term real)
        {"name": "batch_hea", "kind": "batch", "ansatz": "hea", "n": 14, "depth": 10, "sets": 1024,
         "mixed": 64, "each": 4, "lo": 8, "hi": 16},
        # the same for circuits with complex gates, sizes below one block's shared memory
        {"name": "batch_layered", "kind": "batch", "ansatz": "layered", "n": 11, "depth": 6, "sets": 768,
         "mixed": 24, "each": 8, "lo": 8, "hi": 13},
        # a QAOA training step on MaxCut of a 3-regular graph
        {"name": "qaoa_grad_n22", "kind": "qaoa_grad", "n": 22, "depth": 4, "dtype": "c64", "fuse": 4},
        # time evolution of the transverse-field Ising chain
        {"name": "trotter_n26", "kind": "trotter", "n": 26, "steps": 5, "order": 1, "dtype": "c64"},
        # its energy on a large state
        {"name": "tfim_energy_n29", "kind": "energy", "n": 29, "ham": "tfim", "dtype": "c64"},
        # measuring: a million shots of every qubit, and the marginals of ten
        {"name": "measure_n27", "kind": "measure", "n": 27, "shots": 1000000, "marginal": 10, "dtype": "c64"},
    ]


def draw(rng: random.Random):
    kind = rng.choice(("layered", "qft", "layered", "hea_grad", "layered_grad", "batch", "qaoa_grad",
                       "trotter", "energy", "measure"))
    c128 = rng.random() < 0.3
    dtype = "c128" if c128 else "c64"
    less = 1 if c128 else 0
    if kind == "layered":
        if rng.random() < 0.3:
            return {"kind": kind, "n": rng.randint(8, 20), "depth": rng.randint(3, 20), "dtype": dtype, "fuse": 0}
        return {"kind": kind, "n": rng.randint(10, 28 - 2 * less), "depth": rng.randint(5, 30), "dtype": dtype,
                "fuse": rng.randint(3, 5)}
    if kind == "qft":
        return {"kind": kind, "n": rng.randint(12, 29 - 3 * less), "dtype": dtype, "fuse": rng.choice((0, 0, 4))}
    if kind == "hea_grad":
        return {"kind": kind, "n": rng.randint(12, 22 - less), "depth": rng.randint(3, 12), "dtype": dtype,
                "fuse": rng.choice((0, 4, 4))}
    if kind == "layered_grad":
        return {"kind": kind, "n": rng.randint(14, 26 - 2 * less), "depth": rng.randint(4, 12),
                "every": rng.choice((0, 3, 4)), "dtype": dtype, "fuse": rng.choice((3, 4, 4))}
    if kind == "batch":
        if rng.random() < 0.5:
            return {"kind": kind, "ansatz": "hea", "n": rng.randint(8, 14), "depth": rng.randint(4, 10),
                    "sets": rng.randint(64, 1024), "mixed": rng.randint(0, 48), "each": rng.randint(1, 4),
                    "lo": 8, "hi": 16}
        return {"kind": kind, "ansatz": "layered", "n": rng.randint(7, 13), "depth": rng.randint(2, 6),
                "sets": rng.randint(64, 768), "mixed": rng.randint(0, 24), "each": rng.randint(1, 8),
                "lo": 7, "hi": 13}
    if kind == "qaoa_grad":
        return {"kind": kind, "n": 2 * rng.randint(7, 11), "depth": rng.randint(1, 5), "dtype": dtype,
                "fuse": rng.choice((0, 4, 4))}
    if kind == "trotter":
        return {"kind": kind, "n": rng.randint(10, 26 - less), "steps": rng.randint(1, 10),
                "order": rng.randint(1, 2), "dtype": dtype}
    if kind == "energy":
        ham = rng.choice(("tfim", "tfim", "sum_z", "local"))
        return {"kind": kind, "n": rng.randint(10, 24 if ham == "local" else 29 - 2 * less), "ham": ham,
                "dtype": dtype}
    n = rng.randint(12, 27 - 2 * less)
    return {"kind": kind, "n": n, "shots": int(10 ** rng.uniform(2, 6)), "marginal": rng.randint(1, 12),
            "dtype": dtype}


# ---- circuits and Hamiltonians -------------------------------------------------------------
def _gate(kind, targets, controls=(), param=-1, angle=0.0, paulis=""):
    return SimpleNamespace(kind=kind, targets=targets, controls=controls, param=param, angle=angle, paulis=paulis)


def _circuit(n, gates, n_params):
    return SimpleNamespace(n_qubits=n, gates=gates, n_params=n_params)


def _layered(n, depth):
    """RX, RY, RZ on every qubit, then CZ on alternating neighbour pairs, per layer."""
    gates, p = [], 0
    for layer in range(depth):
        for q in range(n):
            for kind in ("RX", "RY", "RZ"):
                gates.append(_gate(kind, (q,), (), p))
                p += 1
        gates += [_gate("Z", (i + 1,), (i,)) for i in range(layer % 2, n - 1, 2)]
    return _circuit(n, gates, p)


def _hea(n, depth):
    """RY on every qubit, then a CZ ladder, per layer."""
    gates = []
    for layer in range(depth):
        gates += [_gate("RY", (q,), (), layer * n + q) for q in range(n)]
        gates += [_gate("Z", (i + 1,), (i,)) for i in range(n - 1)]
    return _circuit(n, gates, n * depth)


def _qft(n):
    gates = []
    for i in range(n):
        gates.append(_gate("H", (i,)))
        gates += [_gate("U1", (i,), (j,), -1, math.pi / (1 << (j - i))) for j in range(i + 1, n)]
    gates += [_gate("SWAP", (i, n - 1 - i)) for i in range(n // 2)]
    return _circuit(n, gates, 0)


def _regular_graph(n, seed):
    """A 3-regular simple graph: half-edges paired at random until no loop or repeat remains."""
    r = random.Random(seed)
    while True:
        stubs = [v for v in range(n) for _ in range(3)]
        r.shuffle(stubs)
        edges = {(min(a, b), max(a, b)) for a, b in zip(stubs[0::2], stubs[1::2])}
        if len(edges) == 3 * n // 2 and all(a != b for a, b in edges):
            return sorted(edges)


def _qaoa(n, edges, p):
    gates = [_gate("H", (q,)) for q in range(n)]
    for layer in range(p):
        gates += [_gate("PAULI", e, (), 2 * layer, paulis="ZZ") for e in edges]
        gates += [_gate("PAULI", (q,), (), 2 * layer + 1, paulis="X") for q in range(n)]
    return _circuit(n, gates, 2 * p)


def _tfim(n):
    return ([(1.0, ((i, "Z"), (i + 1, "Z"))) for i in range(n - 1)]
            + [(0.7, ((i, "X"),)) for i in range(n)])


def _sum_z(n):
    return [(1.0, ((i, "Z"),)) for i in range(n)]


def _maxcut(edges):
    return [(0.5 * len(edges), ())] + [(-0.5, ((i, "Z"), (j, "Z"))) for i, j in edges]


def _local(n, seed):
    """Random strings of one to four letters, two per qubit, as in a chemistry or spin-glass model."""
    r = random.Random(seed)
    terms = []
    for _ in range(2 * n):
        qs = sorted(r.sample(range(n), r.randint(1, 4)))
        terms.append((r.uniform(-1, 1), tuple((q, r.choice("XYZ")) for q in qs)))
    return terms


def _angles(count, seed):
    return np.random.RandomState(seed % (1 << 32)).uniform(0, 2 * math.pi, max(1, count))[:count]


def _terms(case, seed):
    n = case["n"]
    return _tfim(n) if case["ham"] == "tfim" else _sum_z(n) if case["ham"] == "sum_z" else _local(n, seed)


def _amplitudes(n, dtype, seed):
    """A product state of random single-qubit states, disturbed by noise: correlated outcomes and
    energies of order one, as a variational state has."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    a = _angles(2 * n, seed)
    psi = torch.ones(1, dtype=dtype, device="cuda")
    for q in range(n):
        pair = torch.tensor([math.cos(a[2 * q] / 4), math.sin(a[2 * q] / 4) * complex(math.cos(a[2 * q + 1]),
                                                                                      math.sin(a[2 * q + 1]))],
                            dtype=dtype, device="cuda")
        psi = (psi[:, None] * pair[None, :]).reshape(-1)
    psi.add_(torch.randn(1 << n, dtype=dtype, device="cuda", generator=g), alpha=0.3 * 2.0 ** (-n / 2))
    real = torch.view_as_real(psi).reshape(-1)
    parts = real.reshape(-1, min(real.numel(), 1 << 12)).square().sum(1, dtype=torch.float64)
    return psi.mul_(1.0 / math.sqrt(float(parts.sum())))


def _torch_dtype(case):
    return torch.complex64 if case["dtype"] == "c64" else torch.complex128


# ---- what a program holds, and one pass -------------------------------------------------------
def _batch_parts(case, seed):
    """Circuits, items (a circuit index each) and angles of a batch; only the angles follow the seed."""
    make = _hea if case["ansatz"] == "hea" else _layered
    r = random.Random(case["mixed"])
    shapes = [(case["n"], case["depth"])]
    for _ in range(case["mixed"]):
        shapes.append((r.randint(case["lo"], case["hi"]), r.randint(2, case["depth"])))
    circuits = [make(n, d) for n, d in shapes]
    items = [0] * case["sets"] + [1 + i for i in range(case["mixed"]) for _ in range(case["each"])]
    theta = _angles(sum(circuits[i].n_params for i in items), seed)
    return circuits, items, theta


def _grad_parts(case, seed):
    """Circuit, Hamiltonian terms and checkpoint gates of a gradient case."""
    n, depth = case["n"], case["depth"]
    if case["kind"] == "hea_grad":
        return _hea(n, depth), _tfim(n), ()
    if case["kind"] == "qaoa_grad":
        edges = _regular_graph(n, seed)
        return _qaoa(n, edges, depth), _maxcut(edges), ()
    marks, at = [], 0
    for layer in range(depth):
        if case["every"] and layer and layer % case["every"] == 0:
            marks.append(at)
        at += 3 * n + len(range(layer % 2, n - 1, 2))
    return _layered(n, depth), _sum_z(n), tuple(marks)


def _basis(case, seed):
    return random.Random(seed).randrange(1 << case["n"])


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case)
    if kind == "batch":
        circuits, items, theta = _batch_parts(case, seed)
        s.batch = Batch(circuits, [_tfim(c.n_qubits) for c in circuits], items)
        s.theta = torch.from_numpy(theta).cuda()
        return s
    n = case["n"]
    s.state = State(n, case["dtype"])
    if kind == "layered":
        c = _layered(n, case["depth"])
        s.circuit, s.theta = pack_circuit(c), _angles(c.n_params, seed)
    elif kind == "qft":
        s.circuit, s.basis = pack_circuit(_qft(n)), _basis(case, seed)
    elif kind in ("hea_grad", "layered_grad", "qaoa_grad"):
        c, terms, s.marks = _grad_parts(case, seed)
        s.circuit, s.terms = pack_circuit(c), pack_pauli(terms, n)
        s.theta = _angles(c.n_params, seed)
        if kind == "hea_grad":
            s.theta = torch.tensor(s.theta, dtype=torch.float32 if case["dtype"] == "c64" else torch.float64,
                                   device="cuda", requires_grad=True)
    elif kind == "trotter":
        s.terms = pack_pauli(_tfim(n), n)
        s.basis, s.t = _basis(case, seed), 0.1 * case["steps"] * (1 + seed % 7 / 10)
    else:
        s.state.tensor.copy_(_amplitudes(n, _torch_dtype(case), seed))
        if kind == "energy":
            s.terms = pack_pauli(_terms(case, seed), n)
        else:
            s.uniforms = np.random.RandomState(seed % (1 << 32)).random_sample(case["shots"])
    return s


def _as_float(case, value):
    """An energy or gradients, in the precision that the state's type carries."""
    return np.asarray(value, np.float32 if case["dtype"] == "c64" else np.float64)


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "batch":
        e, g = s.batch.run(s.theta)
        return {"energy": e.float(), "grad": g.float()}
    if kind == "layered":
        s.state.init(0).apply_circuit(s.circuit, s.theta, case["fuse"])
        return s.state.tensor
    if kind == "qft":
        s.state.init(s.basis).apply_circuit(s.circuit, None, case["fuse"])
        return s.state.tensor
    if kind == "hea_grad":
        s.theta.grad = None
        e = energy(s.theta, s.state, s.circuit, s.terms, fuse_k=case["fuse"])
        e.backward()
        return {"energy": e.detach().to(s.theta.dtype), "grad": s.theta.grad}
    if kind in ("layered_grad", "qaoa_grad"):
        s.state.init(0)
        e, g = s.state.grad(s.circuit, s.theta, s.terms, s.marks, case["fuse"])
        return {"energy": _as_float(case, e), "grad": _as_float(case, g), "state": s.state.tensor}
    if kind == "trotter":
        s.state.init(s.basis).trotter(s.terms, s.t, case["steps"], case["order"])
        return s.state.tensor
    if kind == "energy":
        return _as_float(case, s.state.expval(s.terms))
    shots = s.state.sample(range(case["n"]), s.uniforms)
    return {"shots": shots.view(np.int64), "marginal": s.state.probabilities(range(case["marginal"]))}


# ---- what a pass cannot do without ---------------------------------------------------------
def _per_gate_bytes(circuit, size):
    """One kernel per gate: every amplitude that a gate changes is read and written."""
    total = 0
    for g in circuit.gates:
        part = 1.0 if g.kind in ("H", "RX", "RY", "RZ") else 0.5
        if g.kind in ("U1", "Z"):
            part = 0.5 ** (1 + len(g.controls))
        total += 2 * size * part
    return total


def work(case):
    kind = case["kind"]
    if kind == "batch":
        bytes_, flops = 0.0, 0.0
        circuits, items, _ = _batch_parts(case, 0)
        for i in items:  # a rotation (6 or 14 flops per amplitude) forward, its inverse on two states
            c = circuits[i]
            flops += (1 << c.n_qubits) * (3 * (6 if case["ansatz"] == "hea" else 14) + 4) * c.n_params
            bytes_ += 8 + 16 * c.n_params
        return {"bytes": bytes_, "flops": flops}
    n = case["n"]
    dim = float(1 << n)
    size = dim * (8 if case["dtype"] == "c64" else 16)
    if kind in ("layered", "qft"):
        c = _qft(n) if kind == "qft" else _layered(n, case["depth"])
        # a merged 1-qubit gate is 14 flops per amplitude, a controlled phase 6 on a quarter
        flops = dim * (1.5 * n * n / 2 + 4 * n if kind == "qft" else 14 * n * case["depth"])
        return {"bytes": size if case["fuse"] else size + _per_gate_bytes(c, size), "flops": flops}
    if kind in ("hea_grad", "layered_grad", "qaoa_grad"):
        per = {"hea_grad": 6 * n, "layered_grad": 14 * n, "qaoa_grad": 6 * n + 6}[kind]
        count = {"hea_grad": n, "layered_grad": 3 * n, "qaoa_grad": n + 1}[kind]
        # forward, the inverse on two states, and an inner product per parameterised gate
        return {"bytes": 2 * size, "flops": dim * case["depth"] * (3 * per + 4 * count)}
    if kind == "trotter":
        return {"bytes": size, "flops": dim * case["steps"] * case["order"] * (6 * n + 6)}
    if kind == "energy":
        return {"bytes": size, "flops": dim * (3 + (4 * n if case["ham"] == "tfim" else 2 * n))}
    return {"bytes": 2 * size + 16.0 * case["shots"], "flops": 4 * dim}


# ---- the same in 64 bits with plain torch -------------------------------------------------------
_ROOT = 1 / math.sqrt(2)


def _matrix(kind, a):
    c, s = math.cos(a / 2), math.sin(a / 2)
    return {"H": ((_ROOT, _ROOT), (_ROOT, -_ROOT)), "RX": ((c, -1j * s), (-1j * s, c)), "RY": ((c, -s), (s, c)),
            "RZ": ((complex(c, -s), 0), (0, complex(c, s)))}[kind]


def _times(x, y):
    return tuple(tuple(sum(x[i][k] * y[k][j] for k in range(2)) for j in range(2)) for i in range(2))


def _split(psi, n, q):
    """The state (..., 2^n) as two halves by qubit q (views)."""
    v = psi.reshape(*psi.shape[:-1], 1 << q, 2, 1 << (n - 1 - q))
    return v[..., 0, :], v[..., 1, :]


def _apply(psi, n, q, m):
    a, b = _split(psi, n, q)
    (m00, m01), (m10, m11) = m
    na = m00 * a
    na.add_(b * m01)
    nb = m10 * a
    nb.add_(b * m11)
    a.copy_(na)
    b.copy_(nb)


def _flip_sign(psi, n, i, j):
    """CZ on neighbours or any two qubits i < j."""
    v = psi.reshape(*psi.shape[:-1], 1 << i, 2, 1 << (j - i - 1), 2, 1 << (n - 1 - j))
    v[..., :, 1, :, 1, :] *= -1


def _letter(psi, n, q, letter):
    """The letter's Pauli matrix on qubit q, in place."""
    a, b = _split(psi, n, q)
    if letter == "Z":
        b.neg_()
        return
    t = a.clone()
    a.copy_(b if letter == "X" else b * -1j)
    b.copy_(t if letter == "X" else t * 1j)


def _string(psi, n, ops):
    out = psi.clone()
    for q, letter in ops:
        _letter(out, n, q, letter)
    return out


def _inner(x, y):
    """<x|y> over the last dimension."""
    return (x.conj() * y).sum(-1)


def _one_letter(lam, psi, n, q, letter):
    """<lam|P|psi> over the last dimension for one letter, without a copy of the state."""
    la, lb = _split(lam, n, q)
    a, b = _split(psi, n, q)
    dot = lambda u, v: (u.conj() * v).sum((-2, -1))  # noqa: E731
    if letter == "Z":
        return dot(la, a) - dot(lb, b)
    if letter == "X":
        return dot(la, b) + dot(lb, a)
    return 1j * (dot(lb, a) - dot(la, b))


def _sum_energy(psi, n, terms):
    total = 0.0
    for c, ops in terms:
        if len(ops) == 1:
            total = total + c * _one_letter(psi, psi, n, *ops[0]).real
        else:
            total = total + c * _inner(psi, _string(psi, n, ops)).real
    return total


def _sum_times(psi, n, terms):
    out = torch.zeros_like(psi)
    for c, ops in terms:
        out.add_(_string(psi, n, ops), alpha=c)
    return out


def _zero(n, rows=0):
    psi = torch.zeros((rows, 1 << n) if rows else (1 << n,), dtype=torch.complex128, device="cuda")
    psi[..., 0] = 1
    return psi


def _forward(psi, n, gates, theta):
    """The gates in order, runs of rotations on one qubit multiplied first."""
    pending = {}
    for g in gates:
        if g.kind in ("Z", "PAULI") and len(g.targets) + len(g.controls) > 1:
            for q in (*g.targets, *g.controls):
                if q in pending:
                    _apply(psi, n, q, pending.pop(q))
            if g.kind == "Z":
                _flip_sign(psi, n, *sorted((*g.targets, *g.controls)))
            else:
                a = theta[g.param]
                t = _string(psi, n, [(q, "Z") for q in g.targets])
                psi.mul_(math.cos(a / 2)).add_(t, alpha=-1j * math.sin(a / 2))
        else:
            kind = "RX" if g.kind == "PAULI" else g.kind
            q, m = g.targets[0], _matrix(kind, theta[g.param] if g.param >= 0 else g.angle)
            pending[q] = _times(m, pending[q]) if q in pending else m
    for q, m in pending.items():
        _apply(psi, n, q, m)


def _gradient(psi, lam, n, gates, theta, count):
    """Reverse sweep: dE/dtheta of every parameter."""
    grad = [0.0] * count
    parts = [[] for _ in range(count)]
    for g in reversed(gates):
        if g.kind == "Z":
            for v in (psi, lam):
                _flip_sign(v, n, *sorted((*g.targets, *g.controls)))
            continue
        if g.kind == "H":
            continue  # only the first layer of a QAOA circuit, before any parameter
        a = theta[g.param]
        if len(g.targets) == 1:
            letter = "X" if g.kind == "PAULI" else g.kind[1]
            parts[g.param].append(_one_letter(lam, psi, n, g.targets[0], letter).imag)
            for v in (psi, lam):
                _apply(v, n, g.targets[0], _matrix("R" + letter, -a))
        else:
            t = _string(psi, n, [(q, "Z") for q in g.targets])
            parts[g.param].append(_inner(lam, t).imag)
            psi.mul_(math.cos(a / 2)).add_(t, alpha=1j * math.sin(a / 2))
            t = _string(lam, n, [(q, "Z") for q in g.targets])
            lam.mul_(math.cos(a / 2)).add_(t, alpha=1j * math.sin(a / 2))
    for p, found in enumerate(parts):
        grad[p] = float(sum(found)) if found else 0.0
    return np.array(grad)


def _exact_batch(case, seed):
    circuits, items, theta = _batch_parts(case, seed)
    offsets = np.concatenate([[0], np.cumsum([circuits[i].n_params for i in items])])
    energies, grads = np.zeros(len(items)), np.zeros(max(1, len(theta)))
    for k, c in enumerate(circuits):
        rows = [j for j, i in enumerate(items) if i == k]
        if not rows:
            continue
        n, terms = c.n_qubits, _tfim(c.n_qubits)
        angle = torch.from_numpy(np.stack([theta[offsets[j]:offsets[j + 1]] for j in rows])).cuda()
        cos = torch.cos(angle / 2).to(torch.complex128)[:, :, None, None]
        sin = torch.sin(angle / 2).to(torch.complex128)[:, :, None, None]

        def matrix(g, sign):
            x, y = cos[:, g.param], sign * sin[:, g.param]
            return {"RX": ((x, -1j * y), (-1j * y, x)), "RY": ((x, -y), (y, x)),
                    "RZ": ((x - 1j * y, 0 * x), (0 * x, x + 1j * y))}[g.kind]

        psi = _zero(n, len(rows))
        for g in c.gates:
            if g.kind == "Z":
                _flip_sign(psi, n, *sorted((*g.targets, *g.controls)))
            else:
                _apply(psi, n, g.targets[0], matrix(g, 1))
        lam = _sum_times(psi, n, terms)
        energies[rows] = _inner(psi, lam).real.cpu().numpy()
        out = torch.zeros(angle.shape, dtype=torch.float64, device="cuda")
        for g in reversed(c.gates):
            if g.kind == "Z":
                for v in (psi, lam):
                    _flip_sign(v, n, *sorted((*g.targets, *g.controls)))
                continue
            out[:, g.param] = _one_letter(lam, psi, n, g.targets[0], g.kind[1]).imag
            for v in (psi, lam):
                _apply(v, n, g.targets[0], matrix(g, -1))
        for row, j in zip(out.cpu().numpy(), rows):
            grads[offsets[j]:offsets[j + 1]] = row
    return {"energy": energies, "grad": grads}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _exact_batch(case, seed)
    n = case["n"]
    if kind == "qft":
        x, dim, out = _basis(case, seed), 1 << n, torch.empty(1 << n, dtype=torch.complex128, device="cuda")
        step = min(dim, 1 << 26)
        for at in range(0, dim, step):
            y = torch.arange(at, at + step, dtype=torch.int64, device="cuda")
            phase = ((y * x) & (dim - 1)).double() * (2 * math.pi / dim)
            out[at:at + step] = torch.polar(torch.full_like(phase, 2.0 ** (-n / 2)), phase)
        return out
    if kind == "layered":
        c, psi = _layered(n, case["depth"]), _zero(n)
        _forward(psi, n, c.gates, _angles(c.n_params, seed))
        return psi
    if kind in ("hea_grad", "layered_grad", "qaoa_grad"):
        c, terms, _ = _grad_parts(case, seed)
        theta = _angles(c.n_params, seed)
        if kind == "hea_grad" and case["dtype"] == "c64":
            theta = theta.astype(np.float32).astype(np.float64)
        psi = _zero(n)
        _forward(psi, n, c.gates, theta)
        final = psi.clone()
        lam = _sum_times(psi, n, terms)
        e = float(_inner(psi, lam).real)
        got = {"energy": np.asarray(e), "grad": _gradient(psi, lam, n, c.gates, theta, c.n_params)}
        if kind != "hea_grad":
            got["state"] = final
        return got
    if kind == "trotter":
        psi, dt = _zero(n), 0.1 * (1 + seed % 7 / 10)
        psi[0] = 0
        psi[_basis(case, seed)] = 1
        half = 2 if case["order"] == 2 else 1
        terms = _tfim(n)
        once = terms if half == 1 else terms + terms[::-1]
        for _ in range(case["steps"]):
            for c, ops in once:
                a = c * dt / half
                if len(ops) == 1:
                    _apply(psi, n, ops[0][0], _matrix("RX", 2 * a))
                else:
                    t = _string(psi, n, ops)
                    psi.mul_(math.cos(a)).add_(t, alpha=-1j * math.sin(a))
        return psi
    psi = _amplitudes(n, _torch_dtype(case), seed).to(torch.complex128)
    if kind == "energy":
        return np.asarray(float(_sum_energy(psi, n, _terms(case, seed))))
    m = case["marginal"]
    p = psi.real.square().add_(psi.imag.square()).reshape(1 << m, -1).sum(1)
    return {"shots": None, "marginal": p / 1.0}
