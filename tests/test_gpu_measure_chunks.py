"""Sampling and probabilities at the edges of their chunks and of the fast
squaring (amplitudes of 2^-5 and more, below 2^-37, zero), bit for bit against
the oracle's exact arithmetic."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_helpers import NP_DTYPE, oracle_threads, rounded

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _state(n, dtype, seed):
    """Amplitudes over many magnitudes: a few dominate, many are tiny or zero."""
    psi = W.random_state(n, seed)
    u = W.uniform_block(seed + 1, 0, 1 << n)
    psi = psi * np.exp2(-60.0 * u ** 3) * (W.uniform_block(seed + 2, 0, 1 << n) > 0.1)
    psi[(1 << n) // 3] = 1.0
    return rounded((psi / np.linalg.norm(psi)).astype(NP_DTYPE[dtype]), dtype)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 6, 7, 8, 11, 17, 18, 20])
def test_samples_and_marginals(n, dtype):
    from paper_2202_07017_gb300 import State
    oracle_threads()
    psi = _state(n, dtype, 40 + n)
    u = W.uniform_block(7, 0, 3000)
    u[:4] = [0.0, 0.5, np.nextafter(1.0, 0.0), 1e-300]
    st = State(n, dtype, guarded=True).load(psi)
    try:
        got = st.sample(range(n), u)
        some = [q for q in range(n) if q % 3 != 1]
        prob = [st.probabilities(qs) for qs in ([0], some[:10], [n - 1], list(range(n))[::-1][:12])]
        st.check_guards()
    finally:
        st.close()
    assert np.array_equal(got, oracle.sample_exact(psi, list(range(n)), u))
    for qs, p in zip(([0], some[:10], [n - 1], list(range(n))[::-1][:12]), prob):
        ref = oracle.probabilities(psi, qs)
        assert np.max(np.abs(p - ref)) <= 1e-12
