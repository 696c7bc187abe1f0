"""Runs of commuting diagonal rotations in one pass and runs of single-qubit
rotations as fused passes: the sizes at which the tiles begin and the launches
split, against the oracle; gradients of such runs against the gate-by-gate
sweep (itself tested against the oracle's shift rule)."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import TOL, gpu_run, max_err, oracle_threads, rounded

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _strings(n, count, seed):
    """`count` random Z strings on 1..n qubits with angles over many turns."""
    rng = W.SplitMix64(seed)
    terms = []
    for _ in range(count):
        ops = tuple((q, "Z") for q in range(n) if rng.next() % 3 == 0) or ((0, "Z"),)
        terms.append((40.0 * (rng.uniform() - 0.5), ops))
    return terms


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,count,order", [(8, 20, 1), (9, 20, 1), (10, 300, 2), (13, 5, 2), (17, 257, 1)])
def test_trotter_of_diagonal_and_single_qubit_terms(n, count, order, dtype):
    from paper_2202_07017_gb300 import State
    oracle_threads()
    terms = _strings(n, count, 70 + n)
    terms += [(0.7 - 0.1 * q, ((q, "XY"[q % 2]),)) for q in range(n)]
    terms += [(0.3, ((0, "X"), (n - 1, "Y")))]
    psi0 = rounded(W.random_state(n, 71), dtype)
    st = State(n, dtype, guarded=True).load(psi0)
    try:
        st.trotter(terms, 0.5, 3, order)
        st.check_guards()
        got = st.numpy()
    finally:
        st.close()
    assert max_err(got, oracle.trotter(psi0, terms, 0.5, 3, order)) <= TOL[dtype]


def _edges_circuit(n, per_layer, params, seed):
    """H, then layers of `per_layer` ZZ / Z / ZZZ rotations sharing `params`
    parameters (every seventh a fixed angle) and an X mixer."""
    rng = W.SplitMix64(seed)
    gates = [W.Gate("H", (q,)) for q in range(n)]
    for layer in range(2):
        for i in range(per_layer):
            k = 2 + rng.next() % 2
            qs = []
            while len(qs) < k:
                q = int(rng.next() % n)
                if q not in qs:
                    qs.append(q)
            p = -1 if i % 7 == 6 else layer * params + int(rng.next() % params)
            gates.append(W.Gate("PAULI", tuple(qs), (), p, 0.3, paulis="Z" * k))
        gates += [W.Gate("PAULI", (q,), (), 2 * params, paulis="X") for q in range(n)]
    theta = np.array([rng.angle() for _ in range(2 * params + 1)])
    return W.Circuit(n, gates, 2 * params + 1), theta


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,per_layer,params", [(10, 3, 3), (10, 150, 140), (12, 140, 2), (17, 40, 7)])
def test_gradients_of_diagonal_runs(n, per_layer, params, dtype):
    from paper_2202_07017_gb300 import State
    oracle_threads()
    c, theta = _edges_circuit(n, per_layer, params, 80 + n)
    terms = W.tfim(n)
    got = gpu_run(c, theta, None, dtype, 4)
    assert max_err(got, oracle.run(c, theta)) <= TOL[dtype]
    res = []
    for fuse_k in (0, 4):
        st = State(n, dtype)
        try:
            res.append(st.init(0).grad(c, theta, terms, (), fuse_k))
        finally:
            st.close()
    (e0, g0), (e1, g1) = res
    bar = {"c64": 1e-5, "c128": 1e-10}[dtype]
    assert abs(e0 - e1) <= bar * sum(abs(k) for k, _ in terms)
    assert np.max(np.abs(g0 - g1)) <= bar * max(1.0, np.max(np.abs(g0)))


def test_angles_without_a_fixed_point_form():
    """A non-finite angle still gives non-finite amplitudes, not an error."""
    from paper_2202_07017_gb300 import State
    c = W.Circuit(10, [W.Gate("PAULI", (0, 3), (), 0, paulis="ZZ")], 1)
    st = State(10, "c64").init(0)
    try:
        st.apply_circuit(c, np.array([np.nan]), 4)
        assert np.isnan(st.numpy()[0])
    finally:
        st.close()
