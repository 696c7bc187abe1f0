"""Complex128 passes: the norm of a state stays within the roundings of its layers'
diagonals."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _norm2(psi):
    v = psi.astype(np.clongdouble)
    return np.sum(v.real**2 + v.imag**2)


@pytest.mark.parametrize("n,fuse_k", [(12, 4), (13, 3), (14, 4)])
def test_norm_of_layered_circuits(n, fuse_k):
    """At most 4 register groups, and so 4 diagonals of 2^-53, a circuit layer, their
    errors independent; an amplitude's own roundings average out."""
    from paper_2202_07017_gb300 import State
    depth, errors = 15, []
    st = State(n, "c128", guarded=True)
    try:
        for seed in range(8):
            c, theta = W.random_layered(n, depth, 60 + seed)
            errors.append(float(_norm2(st.init(0).apply_circuit(c, theta, fuse_k).numpy()) - 1))
        st.check_guards()
    finally:
        st.close()
    assert np.sqrt(np.mean(np.square(errors))) <= 2.0**-53 * np.sqrt((5 if fuse_k == 3 else 4) * depth)

