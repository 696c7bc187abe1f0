"""Complex128 Pauli-string rotations as shears: every number of Y factors modulo 4, angles
in every quarter turn and on their borders, runs of as many diagonal strings as go one
after the other and one more; gradients gate by gate against the oracle's shift rule."""
import math

import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import TOL, max_err, oracle_threads, rounded

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ANGLES = [0.3, math.pi / 4, math.pi / 2, 2.0, math.pi, -math.pi / 2, -2.6, 5 * math.pi / 4, 40.0]
STRINGS = ["ZIZ", "XII", "YII", "XYI", "YYZ", "YYY", "ZXY", "IIZ", "YZX"]


@pytest.mark.parametrize("n", [3, 8, 13])
def test_rotations(n):
    from paper_2202_07017_gb300 import State
    oracle_threads()
    psi = rounded(W.random_state(n, 60 + n), "c128")
    st = State(n, "c128", guarded=True).load(psi)
    ref = psi
    try:
        for i, s in enumerate(STRINGS):
            for j, a in enumerate(ANGLES):
                ops = tuple(((q + i + j) % n, c) for q, c in enumerate(s) if c != "I")
                st.pauli_rotation(ops, a)
                ref = oracle.pauli_rotation(ref, ops, a)
        st.check_guards()
        got = st.numpy()
    finally:
        st.close()
    assert max_err(got, ref) <= TOL["c128"]


@pytest.mark.parametrize("count", [1, 2, 12, 13])
@pytest.mark.parametrize("n", [4, 12])
def test_runs_of_strings(n, count):
    from paper_2202_07017_gb300 import State
    oracle_threads()
    terms = [(ANGLES[k % 9] - 0.1 * k, tuple((q, "Z") for q in range(n) if (k + 1) >> (q % 4) & 1))
             for k in range(count)]
    psi = rounded(W.random_state(n, 70 + n), "c128")
    st = State(n, "c128", guarded=True).load(psi)
    try:
        st.trotter(terms, 0.9, 1, 1)
        st.check_guards()
        got = st.numpy()
    finally:
        st.close()
    assert max_err(got, oracle.trotter(psi, terms, 0.9, 1, 1)) <= TOL["c128"]


@pytest.mark.parametrize("n", [3, 7])
def test_gradients(n):
    from paper_2202_07017_gb300 import State
    oracle_threads()
    gates = [W.Gate("RY", (q,), (), -1, 0.4 + q) for q in range(n)]
    for i, s in enumerate(STRINGS):
        qs = [q for q, c in enumerate(s) if c != "I"]
        gates.append(W.Gate("PAULI", tuple((q + i) % n for q in qs), (), i, paulis=s.replace("I", "")))
    c, theta = W.Circuit(n, gates, len(STRINGS)), np.array(ANGLES)
    terms = W.tfim(n)
    st = State(n, "c128").init(0)
    try:
        e, g = st.grad(c, theta, terms)
    finally:
        st.close()
    ref = oracle.grad_param_shift(c, theta, terms)
    assert abs(e - oracle.energy(c, theta, terms)) <= 1e-11
    assert np.max(np.abs(g - ref)) <= 1e-10 * max(1.0, np.max(np.abs(ref)))


@pytest.mark.parametrize("n,layers", [(3, 40), (12, 12)])
def test_complex64_keeps_the_norm(n, layers):
    """One angle on every edge, many times, forward and back: no scale repeats."""
    from paper_2202_07017_gb300 import State
    oracle_threads()
    gates = [W.Gate("H", (q,)) for q in range(n)]
    for _ in range(layers):
        gates += [W.Gate("PAULI", (q, (q + 1) % n), (), 0, paulis="ZZ") for q in range(n)]
        gates += [W.Gate("PAULI", (q,), (), 1, paulis="X") for q in range(n)]
    c, theta = W.Circuit(n, gates, 2), np.array([0.7, 2.2])
    terms = W.tfim(n)
    st = State(n, "c64").init(0)
    try:
        e, g = st.grad(c, theta, terms)
        norm = st.init(0).apply_circuit(c, theta).norm()
    finally:
        st.close()
    ref, count, scale = oracle.grad_param_shift(c, theta, terms), len(gates), sum(t[0] for t in terms)
    # a rotation's rounding is a fraction of 2^-24 of random sign on each of `count` gates;
    # a repeated scale would be up to 2^-24 times all of them
    bar = 4 * math.sqrt(count) * 2.0 ** -24
    assert abs(norm - 1) <= bar
    assert abs(e - oracle.energy(c, theta, terms)) <= bar * scale
    assert np.max(np.abs(g - ref)) <= bar * scale * layers * n
