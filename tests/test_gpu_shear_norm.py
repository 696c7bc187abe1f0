"""Complex64 Pauli rotations gate by gate, one angle hundreds of times: neither the norm
nor a gradient takes on a scale that the rounded sine and cosine would repeat."""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HALF = 0.745  # fl32(cos)^2 + fl32(sin)^2 = 1 + 8.2e-8
N, COUNT = 6, 600
BAR = 4 * math.sqrt(COUNT) * 2.0**-24  # roundings of random sign on each gate: 5.8e-6


def test_the_angle_shows_a_repeated_scale():
    c, s = (float(np.float32(f(HALF))) for f in (math.cos, math.sin))
    assert COUNT * abs(c * c + s * s - 1) > 8 * BAR


@pytest.mark.parametrize("letters", ["ZZ", "XY"])
def test_one_angle_on_many_strings(letters):
    from paper_2202_07017_gb300 import State
    gates = [W.Gate("RY", (q,), (), -1, 0.4 + q) for q in range(N)]
    gates += [W.Gate("PAULI", (k % N, (k + 1) % N), (), k, paulis=letters) for k in range(COUNT)]
    c, theta, terms = W.Circuit(N, gates, COUNT), np.full(COUNT, 2 * HALF), [(1.0, ((q, "X"),)) for q in range(N)]
    got = {}
    for dtype in ("c64", "c128"):
        st = State(N, dtype, guarded=True)
        try:
            got[dtype] = st.init(0).grad(c, theta, terms, (), 0)
            norm = st.init(0).apply_circuit(c, theta).norm()
            st.check_guards()
        finally:
            st.close()
        if dtype == "c64" and letters == "ZZ":
            assert abs(norm - 1) <= BAR
    (e, g), (e0, g0) = got["c64"], got["c128"]
    if letters == "ZZ":
        assert abs(e - e0) <= BAR * N
        # forward and back: twice the gates
        assert np.max(np.abs(g - g0)) <= 2 * BAR * N
    else:  # forward by products with the feedback; the way back keeps both states' scale
        assert np.max(np.abs(g - g0)) <= 4 * BAR * N
