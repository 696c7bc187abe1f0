"""Fused passes on planes (complex64, states of 20 qubits and more) at the
edges of their layout: groups with and without amplitude bit 0, layers that
rotate some or all bits, real and complex diagonals, angles at which the
rotation's form changes, against the oracle."""
import math

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import TOL, gpu_run, max_err, oracle_threads, rounded

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,fuse_k", [(20, 4), (21, 4), (21, 5), (22, 4)])
@pytest.mark.parametrize("kinds", [("H", "Z", "U1"), ("RY", "Z"), ("RX", "RY", "RZ", "H", "U1", "Z")])
def test_random_rotations_and_phases(n, fuse_k, kinds):
    """1-qubit gates and phases on random qubits (few per layer and many)."""
    oracle_threads()
    c, theta = W.random_gates(n, 120, 50 + n, max_ctrl=2, kinds=kinds)
    gates = [g for g in c.gates if not g.controls or g.kind in ("Z", "U1")]
    c = W.Circuit(n, gates, c.n_params)
    psi0 = rounded(W.random_state(n, 51), "c64")
    got = gpu_run(c, theta, psi0, "c64", fuse_k)
    assert max_err(got, oracle.run(c, theta, psi0)) <= TOL["c64"]


def test_special_angles_on_the_lowest_qubits():
    """Rotations by multiples of pi / 2 and by small angles on bits 0..4."""
    oracle_threads()
    n = 20
    angles = [0.0, math.pi / 2, math.pi, -math.pi / 2, 2 * math.pi, 1e-4, math.pi - 1e-4, 3.0]
    gates, theta = [], []
    for rep, a in enumerate(angles):
        for q in range(n - 5, n):
            for kind in ("RX", "RY", "RZ")[rep % 3:] + ("RX",):
                gates.append(W.Gate(kind, (q,), (), len(theta)))
                theta.append(a * (1 if q % 2 else -1))
        gates += [W.Gate("Z", (q + 1,), (q,)) for q in range(n - 5, n - 1)]
    c = W.Circuit(n, gates, len(theta))
    psi0 = rounded(W.random_state(n, 52), "c64")
    got = gpu_run(c, np.array(theta), psi0, "c64", 4)
    assert max_err(got, oracle.run(c, np.array(theta), psi0)) <= TOL["c64"]


def _grad_circuit(n, depth, seed):
    """Rotations about one to three axes per qubit and layer in a seeded order, a
    parameter shared by two gates, fixed rotations and Hadamards between them,
    CZs, controlled phases, and one controlled rotation (not a layer program)."""
    rng = W.SplitMix64(seed)
    gates, theta = [], []
    for layer in range(depth):
        for q in range(n):
            for _ in range(1 + rng.next() % 3):
                kind = ("RX", "RY", "RZ", "H")[rng.next() % 4]
                if kind == "H":
                    gates.append(W.Gate("H", (q,)))
                elif theta and rng.next() % 8 == 0:
                    gates.append(W.Gate(kind, (q,), (), len(theta) - 1))
                elif rng.next() % 8 == 0:
                    gates.append(W.Gate(kind, (q,), (), -1, rng.angle()))
                else:
                    theta.append(rng.angle())
                    gates.append(W.Gate(kind, (q,), (), len(theta) - 1))
        gates += [W.Gate("Z", (i + 1,), (i,)) for i in range(layer % 2, n - 1, 2)]
        gates.append(W.Gate("U1", (0,), (n - 1,), -1, rng.angle()))
    theta.append(rng.angle())
    gates.append(W.Gate("RY", (1,), (n - 2,), len(theta) - 1))
    gates += [W.Gate("RX", (q,), (), 0) for q in range(0, n, 3)]
    return W.Circuit(n, gates, len(theta)), np.array(theta)


@pytest.mark.parametrize("n,depth,checks", [(19, 3, 0), (20, 3, 0), (21, 2, 1), (22, 3, 0)])
def test_gradients_on_planes(n, depth, checks):
    """Every gradient against the gate-by-gate sweep, which the oracle's shift
    rule pins elsewhere."""
    from paper_2202_07017_gb300 import State
    c, theta = _grad_circuit(n, depth, 90 + n)
    terms = W.tfim(n)
    marks = [len(c.gates) // 2] if checks else []
    res = []
    for fuse_k in (0, 4):
        st = State(n, "c64", guarded=True)
        try:
            res.append(st.init(0).grad(c, theta, terms, marks, fuse_k))
            st.check_guards()
        finally:
            st.close()
    (e0, g0), (e1, g1) = res
    assert abs(e0 - e1) <= TOL["c64"] * sum(abs(k) for k, _ in terms)
    assert np.max(np.abs(g0 - g1)) <= TOL["c64"] * max(1.0, np.max(np.abs(g0)))
