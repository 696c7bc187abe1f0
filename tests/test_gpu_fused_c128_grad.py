"""Complex128 reverse sweeps in passes: gradients as exact as the gates' own matrices
leave them (no products with phases of other gates in between)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kind", ["RY", "RX"])
def test_gradients_against_the_gate_by_gate_sweep(kind):
    """N rotations forward and N un-applied, each an independent rounding of its matrix of
    about 2^-53: sqrt(2 N) of them, and twice that for the passes' own products."""
    from paper_2202_07017_gb300 import State
    n, depth, errors = 12, 8, []
    one, passes = State(n, "c128"), State(n, "c128", guarded=True)
    try:
        for seed in range(8):
            c, theta = W.hea(n, depth, 300 + seed)
            c = W.Circuit(n, [W.Gate(kind, g.targets, (), g.param) if g.kind == "RY" else g
                              for g in c.gates], c.n_params)
            _, g0 = one.init(0).grad(c, theta, W.tfim(n), (), 0)
            _, g1 = passes.init(0).grad(c, theta, W.tfim(n), (), 4)
            errors.append(np.max(np.abs(g1 - g0)) / np.max(np.abs(g0)))
        passes.check_guards()
    finally:
        one.close()
        passes.close()
    assert np.sqrt(np.mean(np.square(errors))) <= 2 * 2.0**-53 * np.sqrt(2 * n * depth)
