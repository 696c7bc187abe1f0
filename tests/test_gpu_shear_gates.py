"""Complex128 1-qubit gates as shears: angles in every quarter turn and at their
borders, reflections, phases with controls, matrices close to but not unitary
(which keep the products), and their un-applies, against the oracle."""
import math

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import TOL, gpu_run, max_err, oracle_threads, rounded

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ANGLES = [0.0, 1e-9, math.pi / 4, math.pi / 2, math.pi / 2 + 1e-12, 3 * math.pi / 4, math.pi,
          -math.pi / 2, 5 * math.pi / 4, 3 * math.pi / 2, 2 * math.pi, -7.0, 100.0]


@pytest.mark.parametrize("n", [1, 5, 11])
def test_rotations_and_phases(n):
    oracle_threads()
    gates, theta = [], []
    for i, a in enumerate(ANGLES):
        q = i % n
        ctrl = ((q + 1) % n,) if n > 1 and i % 2 else ()
        for kind in ("RX", "RY", "RZ", "U1"):
            if kind == "U1":
                gates.append(W.Gate(kind, (q,), ctrl, -1, a))
            else:
                theta.append(a)
                gates.append(W.Gate(kind, (q,), ctrl, len(theta) - 1))
        gates += [W.Gate(k, (q,), ctrl) for k in ("H", "X", "Y", "Z")]
    c, th = W.Circuit(n, gates, len(theta)), np.array(theta)
    psi0 = rounded(W.random_state(n, 33), "c128")
    assert max_err(gpu_run(c, th, psi0, "c128"), oracle.run(c, th, psi0)) <= TOL["c128"]


@pytest.mark.parametrize("eps", [0.0, 1e-14, 1e-9, 0.3])
def test_matrices_near_rotations(eps):
    """[[c, -s], [s, c]] and its kin scaled by 1 + eps: applied as given."""
    oracle_threads()
    n, c, s = 6, math.cos(0.7), math.sin(0.7)
    mats = [np.array([[c, -s], [s, c]]), np.array([[c, s], [s, -c]]), np.array([[c, 1j * s], [1j * s, c]]),
            np.diag([c + 1j * s, c - 1j * s])]
    gates = [W.Gate("MATRIX", (q,), (), matrix=(1 + eps) * m.astype(complex))
             for q in range(n) for m in mats]
    circ = W.Circuit(n, gates, 0)
    psi0 = rounded(W.random_state(n, 34), "c128")
    ref = oracle.run(circ, None, psi0)
    assert max_err(gpu_run(circ, None, psi0, "c128"), ref) <= TOL["c128"] * np.max(np.abs(ref))


def test_unapplied_gates():
    """Gradients gate by gate (the un-applies as shears) against the oracle's
    exact shift rule."""
    from paper_2202_07017_gb300 import State
    oracle_threads()
    n = 6
    c, theta = W.random_layered(n, 2, 35)
    terms = W.tfim(n)
    st = State(n, "c128").init(0)
    try:
        e, g = st.grad(c, theta, terms)
    finally:
        st.close()
    ref = oracle.grad_param_shift(c, theta, terms)
    assert abs(e - oracle.energy(c, theta, terms)) <= 1e-11
    assert np.max(np.abs(g - ref)) <= 1e-10 * np.max(np.abs(ref))
