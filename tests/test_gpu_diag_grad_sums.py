"""Gradients of many diagonal rotations on one parameter: the terms' sum keeps the
precision of a compensated sum."""
import itertools

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [10, 13])
@pytest.mark.parametrize("flip", [0, 5, 9])
@pytest.mark.parametrize("value", [0.52497673, 0.54937172, 0.92236722, 0.97490299])
def test_equal_terms(n, flip, value):
    """psi = |0...0> + i v |flip>, H = X on that qubit, 127 strings that hold it, all by
    the angle 0 of one parameter: every Im<H psi|P|psi> is -2 v, in exact fp32."""
    from paper_2202_07017_gb300 import State
    v = float(np.float32(value)) / 2
    others = [q for q in range(n) if q != flip]
    sets = [(flip, *s) for k in range(4) for s in itertools.combinations(others, k)][1:128]
    gates = [W.Gate("PAULI", s, (), 0, paulis="Z" * len(s)) for s in sets]
    psi = np.zeros(1 << n, np.complex64)
    psi[0], psi[1 << (n - 1 - flip)] = 1, 1j * v
    st = State(n, "c64", guarded=True)
    try:
        e, g = st.load(psi).grad(W.Circuit(n, gates, 1), np.zeros(1), [(1.0, ((flip, "X"),))], (), 4)
        st.check_guards()
    finally:
        st.close()
    # two roundings of a product, four of a tile's transform, one of a sum, one of the turn
    assert abs(abs(g[0]) - 2 * v * len(gates)) <= 8 * 2.0**-24 * 2 * v * len(gates)
