"""Diagonal MATRIX gates need not be unitary: projectors and other diagonals with
zeros or very small entries inside fused passes, beside rotations whose diagonals
are rounded with feedback, against the oracle; the state stays usable."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import TOL, gpu_run, max_err, oracle_threads, rounded

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (diagonal on a qubit, diagonal under a control)
DIAGONALS = {"upper": ((1, 0), (0, 1)), "lower": ((1, 0), (1, 0)), "scaled": ((1, 0.5j), (0, 0.5 + 0.25j)),
             "tiny": ((1, 1e-40), (1e-40, 1))}


def _check(n, fuse_k, alone, under_control):
    oracle_threads()
    rng = W.SplitMix64(7 * n)
    gates, theta = [], []

    def rotations():
        for q in range(n):
            for kind in ("RX", "RZ", "RY"):
                gates.append(W.Gate(kind, (q,), (), len(theta)))
                theta.append(rng.angle())
        gates.extend(W.Gate("Z", (i + 1,), (i,)) for i in range(n - 1))

    rotations()
    gates.append(W.Gate("MATRIX", (n // 2,), (), matrix=np.diag(np.array(alone, complex))))
    gates.append(W.Gate("MATRIX", (1,), (n - 1,), matrix=np.diag(np.array(under_control, complex))))
    gates.append(W.Gate("RZ", (n // 2,), (), -1, 0.3))
    rotations()
    c = W.Circuit(n, gates, len(theta))
    psi0 = rounded(W.random_state(n, 8), "c64")
    got = gpu_run(c, np.array(theta), psi0, "c64", fuse_k)
    want = oracle.run(c, np.array(theta), psi0)
    assert max_err(got, want) <= TOL["c64"]
    # 13 operations a qubit of at most 4 roundings each, relative to the norm
    assert np.linalg.norm(got - want) <= 13 * n * 4 * 2.0**-24 * np.linalg.norm(want)


@pytest.mark.parametrize("n,fuse_k", [(12, 4), (20, 4), (20, 3), (21, 4)])
@pytest.mark.parametrize("diag", sorted(DIAGONALS))
def test_diagonals_with_zeros(n, fuse_k, diag):
    _check(n, fuse_k, *DIAGONALS[diag])


# matrices that scale the state, as they stand: alone they are applied gate by gate,
# in passes they multiply with the rotations beside them
MATRICES = {"scaled": 0.6 * np.array([[0.8, -0.6], [0.6, 0.8]]), "projector": np.diag([0, 1]),
            "diagonal": np.diag([0.3 + 0.1j, 0.7]), "damping": np.array([[1, 0], [0.1, 0.9]])}


@pytest.mark.parametrize("n,fuse_k", [(6, 0), (12, 4), (20, 4), (20, 3)])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_matrices_that_are_not_unitary(n, fuse_k, name):
    oracle_threads()
    rng = W.SplitMix64(11 * n)
    gates, theta = [], []
    for layer in range(3):
        for q in range(n):
            theta.append(rng.angle())
            gates.append(W.Gate(("RX", "RY", "RZ")[(q + layer) % 3], (q,), (), len(theta) - 1))
        gates += [W.Gate("Z", (i + 1,), (i,)) for i in range(layer % 2, n - 1, 2)]
        for q in (1, n // 2):
            gates.append(W.Gate("MATRIX", (q,), (), matrix=MATRICES[name].astype(complex)))
        gates += [W.Gate("H", (q,)) for q in range(n)]
    c = W.Circuit(n, gates, len(theta))
    psi0 = rounded(W.random_state(n, 9), "c64")
    got = gpu_run(c, np.array(theta), psi0, "c64", fuse_k)
    want = oracle.run(c, np.array(theta), psi0)
    # 12 operations a qubit of at most 4 roundings each, relative to the norm; the state
    # before a projector may be twice as long, three times over
    assert np.linalg.norm(got - want) <= 8 * 12 * n * 4 * 2.0**-24 * np.linalg.norm(want)
