"""Batches of real gates (states as real vectors, rotations as shears, runs of
sign flips as patterns): circuits below, at and above one register tile, angles
past pi, controlled gates between flips on the same qubits, and more sign
patterns than are kept; against the oracle's energies and shift-rule gradients."""
import math

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import oracle_threads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _random_real(n, n_gates, seed):
    rng = W.SplitMix64(seed)
    gates, npar = [], 0
    for _ in range(n_gates):
        q = sorted(range(n), key=lambda _: rng.next())
        kind = ("RY", "Z", "Z", "RY", "H", "X", "Z")[rng.next() % 7]
        ctrl = tuple(q[1:1 + rng.next() % min(3, n)])
        par = -1
        if kind == "RY":
            par, npar = npar, npar + 1
        gates.append(W.Gate(kind, (q[0],), ctrl, par))
    return W.Circuit(n, gates, npar)


def _alternating(n, pairs):
    """CZ and RY in turn on the same qubits: a pattern for every CZ."""
    gates = []
    for i in range(pairs):
        gates += [W.Gate("Z", (i % n,), ((i + 1) % n,)), W.Gate("RY", ((i + 1) % n,), (), i)]
    return W.Circuit(n, gates, pairs)


def _circuits():
    return ([_random_real(n, 60, 40 + n) for n in (1, 2, 4, 5, 6, 9, 10)]
            + [_alternating(5, 40), _alternating(6, 200), W.hea(11, 2, 7)[0]])


@pytest.mark.parametrize("tune", [4, 1], ids=["real", "tuned"])
def test_real_batch(tune):
    from paper_2202_07017_gb300 import Batch
    oracle_threads()
    circuits = _circuits()
    hams = [W.tfim(c.n_qubits) if c.n_qubits > 1 else [(1.0, ((0, "X"),)), (0.5, ((0, "Z"),))]
            for c in circuits]
    rng = np.random.default_rng(5)
    thetas = [rng.uniform(-7, 7, c.n_params) for c in circuits]
    thetas[-1][:4] = [math.pi, -math.pi, 3 * math.pi, 0.0]
    b = Batch(circuits, hams, list(range(len(circuits))), tune=tune)
    e, g = b.run(torch.tensor(np.concatenate(thetas), dtype=torch.float64, device="cuda"))
    e, g, real = e.cpu().numpy(), g.cpu().numpy(), b.real
    b.close()
    assert real or tune == 1
    off = 0
    for i, (c, h, th) in enumerate(zip(circuits, hams, thetas)):
        scale = sum(abs(t[0]) for t in h)
        # 400 gates' fp32 roundings, 400 * 2^-24 relative at the worst
        assert abs(e[i] - oracle.energy(c, th, h)) <= 2.4e-5 * scale, i
        if c.n_params:
            ref = oracle.grad_param_shift(c, th, h)
            assert np.max(np.abs(g[off:off + c.n_params] - ref)) <= 2.4e-5 * scale, i
        off += c.n_params
