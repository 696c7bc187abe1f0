"""Batches over the size classes: teams of 64 to 512 threads side by side, items over four
blocks' shared memory and beyond it, alone and mixed, more of them than clusters;
parameters that several rotations of one group share.  Energies and sampled
gradients against the oracle; equal items give equal results."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import oracle_threads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _layered(n, depth, shared):
    c, th = W.random_layered(n, depth, 7 * n + depth)
    if shared:  # one angle for each kind and layer
        gates = [g if g.param < 0 else W.Gate(g.kind, g.targets, g.controls,
                                              3 * (g.param // (3 * n)) + g.param % 3)
                 for g in c.gates]
        c, th = W.Circuit(n, gates, 3 * depth), th[:3 * depth]
    return c, th


def _hea(n, depth, shared):
    c, th = W.hea(n, depth, 3 * n + depth)
    if shared:
        gates = [g if g.param < 0 else W.Gate(g.kind, g.targets, g.controls, g.param // n)
                 for g in c.gates]
        m = 1 + max(g.param for g in gates)
        c, th = W.Circuit(n, gates, m), th[:m]
    return c, th


def _check(circuits, thetas, items, tune):
    from paper_2202_07017_gb300 import Batch
    oracle_threads()
    hams = [W.tfim(c.n_qubits) for c in circuits]
    b = Batch(circuits, hams, items, tune=tune)
    theta = torch.tensor(np.concatenate([thetas[i] for i in items]), dtype=torch.float64, device="cuda")
    e, g = b.run(theta)
    e2, g2 = b.run(theta, graph=True)
    e, g, e2, g2 = (t.cpu().numpy() for t in (e, g, e2, g2))
    b.close()
    assert np.array_equal(e, e2) and np.array_equal(g, g2)
    first, off = {}, 0
    for k, i in enumerate(items):
        c, h, th = circuits[i], hams[i], thetas[i]
        gi = g[off:off + c.n_params]
        off += c.n_params
        if i in first:
            assert e[k] == e[first[i][0]] and np.array_equal(gi, first[i][1])
            continue
        first[i] = (k, gi)
        scale = sum(abs(t[0]) for t in h)
        bound = len(c.gates) * 2.0 ** -24  # one fp32 rounding a gate, all with one sign
        assert abs(e[k] - oracle.energy(c, th, h)) <= bound * scale, c.n_qubits
        ps = sorted({0, c.n_params // 2, c.n_params - 1})
        ref = oracle.grad_param_shift(c, th, h, params=ps)
        uses = max(np.bincount([q.param for q in c.gates if q.param >= 0]))
        assert np.max(np.abs(gi[ps] - ref[ps])) <= bound * uses * scale, c.n_qubits


@pytest.mark.parametrize("tune", [1, 3], ids=["tuned", "shared"])
def test_complex_sizes(tune):
    parts = [_layered(n, 2 if n < 13 else 1, False) for n in (2, 8, 9, 10, 11, 12, 13, 14, 15, 16)]
    _check([p[0] for p in parts], [p[1] for p in parts], [i for i in range(10) for _ in range(3)], tune)


@pytest.mark.parametrize("tune", [1, 4], ids=["tuned", "real"])
def test_real_sizes(tune):
    parts = [_hea(n, 2, False) for n in (3, 9, 10, 11, 12, 13, 14, 15, 16, 17)]
    _check([p[0] for p in parts], [p[1] for p in parts], [i for i in range(10) for _ in range(3)], tune)


def test_shared_parameters():
    parts = [_hea(n, 2, True) for n in (6, 15)] + [_layered(n, 2, True) for n in (5, 10, 15)]
    _check([p[0] for p in parts], [p[1] for p in parts], [0, 1, 2, 3, 4], 3)


@pytest.mark.parametrize("n,tune", [(16, 4), (15, 3)])
def test_more_wide_items_than_clusters(n, tune):
    c, th = (_hea if tune == 4 else _layered)(n, 1, False)
    _check([c], [th], [0] * 90, tune)
