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
