"""One-kernel-per-gate launches at the sizes where their shape changes (units
per thread 8 -> 4 -> 2 -> 1, then blocks of 256 -> 128 -> 64 threads): random
gates of every kind, with and without controls, against the oracle."""
import pytest

import oracle
import workloads as W
from gpu_helpers import TOL, max_err, oracle_threads, rounded

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 6, 7, 14, 15, 16, 19, 20, 21, 22])
def test_random_gates_over_launch_shapes(n, dtype):
    from paper_2202_07017_gb300 import State
    oracle_threads()
    c, theta = W.random_gates(n, 40 if n < 18 else 24, 900 + n)
    psi0 = rounded(W.random_state(n, 901), dtype)
    st = State(n, dtype, guarded=True)
    try:
        got = st.load(psi0).apply_circuit(c, theta).numpy()
        st.check_guards()
    finally:
        st.close()
    assert max_err(got, oracle.run(c, theta, psi0)) <= TOL[dtype]


def test_captured_circuit_replays():
    """A circuit's launches captured into a CUDA graph and replayed on a fresh
    basis state give the amplitudes of the plain launches."""
    from paper_2202_07017_gb300 import State, pack_circuit
    n = 9
    c, theta = W.random_layered(n, 3, 17)
    pc = pack_circuit(c)
    side = torch.cuda.Stream()
    st = State(n, "c128", stream=side)
    try:
        with torch.cuda.stream(side):
            want = st.init(3).apply_circuit(pc, theta).numpy()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            st.init(3).apply_circuit(pc, theta)
        st.init(0)
        graph.replay()
        torch.cuda.synchronize()
        got = st.numpy()
    finally:
        st.close()
    assert (got == want).all()
