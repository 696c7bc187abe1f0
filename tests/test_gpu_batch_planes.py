"""Batches of complex gates on planes: states narrower than a register tile, at the
sizes where a thread takes eight slices of the terms, in shared and in global memory;
rotations at and past whole turns, controlled kinds between flips, terms with odd
and even numbers of Y; against the oracle's energies and shift-rule gradients."""
import math

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import oracle_threads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ONEQ = ("H", "X", "Y", "Z", "RX", "RY", "RZ", "U1")


@pytest.mark.parametrize("tune", [0, 1, 3], ids=["global", "tuned", "shared"])
def test_complex_batch(tune):
    from paper_2202_07017_gb300 import Batch
    oracle_threads()
    circuits, hams, thetas = [], [], []
    for n in (1, 2, 3, 4, 9, 10, 13):
        c, th = W.random_layered(n, 3 if n < 10 else 1, n)
        th[: 4] = [math.pi, 2 * math.pi, -3 * math.pi, 0.0][: min(4, len(th))]
        circuits.append(c), thetas.append(th)
        hams.append(W.random_pauli_sum(n, min(20, 4 ** n - 1), n))
    for n, ctrl in ((4, 3), (10, 2), (11, 3)):
        c, th = W.random_gates(n, 70, 50 + n, max_tar=1, max_ctrl=ctrl, kinds=ONEQ)
        circuits.append(c), thetas.append(th)
        hams.append(W.random_pauli_sum(n, 24, n))
    b = Batch(circuits, hams, list(range(len(circuits))), tune=tune)
    e, g = b.run(torch.tensor(np.concatenate(thetas), dtype=torch.float64, device="cuda"))
    e, g = e.cpu().numpy(), g.cpu().numpy()
    b.close()
    off = 0
    for i, (c, h, th) in enumerate(zip(circuits, hams, thetas)):
        scale = sum(abs(t[0]) for t in h)
        # up to 120 gates' fp32 roundings, 120 * 2^-24 relative at the worst
        assert abs(e[i] - oracle.energy(c, th, h)) <= 7.2e-6 * scale, i
        if c.n_params:
            ps = sorted({int(p) for p in np.linspace(0, c.n_params - 1, 24)})
            ref = oracle.grad_param_shift(c, th, h, params=ps)
            assert np.max(np.abs(g[off:off + c.n_params][ps] - ref[ps])) <= 7.2e-6 * scale, i
        off += c.n_params
