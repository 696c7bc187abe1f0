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
