"""Runs of X and Y rotations as three shears: each rotation's angle is rounded once
(a fine time evolution repeats the same rotation, and its error, in every step)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("letter", ["X", "Y"])
@pytest.mark.parametrize("n,qubit", [(10, 9), (12, 0), (12, 6), (13, 11)])
def test_one_rotation_among_zeros(n, qubit, letter):
    """exp(-i a X) or exp(-i a Y) on one qubit of |0...0> in a run with zero angles: the
    smaller of sine and cosine is the fp32 number next to it."""
    from paper_2202_07017_gb300 import State
    angles = np.random.RandomState(5).uniform(-math.pi, math.pi, 24)
    st = State(n, "c64", guarded=True)
    try:
        for a in angles:
            terms = [(a if q == qubit else 0.0, ((q, letter),)) for q in range(n)]
            got = st.init(0).trotter(terms, 1.0, 1, 1).numpy()
            st.check_guards()
            c, s = got[0], got[1 << (n - 1 - qubit)]
            s = -s.imag if letter == "X" else s.real
            assert np.count_nonzero(got) == 2
            small, large = sorted(((c.real, math.cos(a)), (s, math.sin(a))), key=lambda v: abs(v[1]))
            assert abs(small[0] - small[1]) <= 0.51 * np.spacing(np.float32(abs(small[1])))
            assert abs(large[0] - large[1]) <= 2.0**-23  # 1 + a b: three roundings
    finally:
        st.close()
