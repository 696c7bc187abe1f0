"""Runs of diagonal Pauli rotations by small angles: the angle of every amplitude
keeps its relative accuracy, as a time evolution in many fine steps needs (an
absolute error would be the same in every step)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _strings(n, k, seed):
    """k distinct diagonal strings of one to four letters."""
    rng = np.random.RandomState(seed)
    seen = []
    while len(seen) < k:
        qs = tuple(sorted(rng.choice(n, rng.randint(1, 5), replace=False)))
        if qs not in seen:
            seen.append(qs)
    return seen


@pytest.mark.parametrize("dtype,k", [("c64", 5), ("c64", 25), ("c64", 257), ("c128", 13), ("c128", 40)])
@pytest.mark.parametrize("size", [1e-9, 1e-6, 1e-4, 1e-2, 0.3])
@pytest.mark.parametrize("equal", [False, True])
def test_angles_of_one_run(dtype, k, size, equal):
    from paper_2202_07017_gb300 import State
    n = 10
    rng = np.random.RandomState(k)
    coeff = size * (np.ones(k) if equal else rng.uniform(-1, 1, k)) * 1.2345678
    strings = _strings(n, k, 3)
    x = np.arange(1 << n)
    total = np.zeros(1 << n, np.longdouble)
    for c, qs in zip(coeff, strings):
        parity = sum((x >> (n - 1 - int(q))) & 1 for q in qs) & 1
        total += np.longdouble(c) * (1 - 2 * parity)
    amp = 2.0 ** (-n / 2)
    st = State(n, dtype, guarded=True)
    try:
        st.load(np.full(1 << n, amp, np.complex64 if dtype == "c64" else np.complex128))
        got = st.trotter([(float(c), tuple((int(q), "Z") for q in qs)) for c, qs in zip(coeff, strings)],
                         1.0, 1, 1).numpy().astype(np.clongdouble) / amp
        st.check_guards()
    finally:
        st.close()
    # the turn and each angle's step (up to 2^-31 of the sum of magnitudes), sine and
    # cosine (2 roundings) and product (2), per launch
    u = 2.0 ** (-24 if dtype == "c64" else -53)
    step = 2.0 ** (-31 if dtype == "c64" else -61)
    launches = -(-k // 256)
    bound = np.abs(coeff).sum() * (k * step + 6 * u) * launches
    assert np.max(np.abs(got.imag + np.sin(total))) <= bound + 2 * u * launches * np.max(np.abs(np.sin(total)))
    assert np.max(np.abs(got.real - np.cos(total))) <= bound + 4 * u * launches
