"""The step calls copy their k-point parameters from two pinned buffers in turn and do not wait for them: calls in quick
succession, with other k-points, batch sizes and lattices each, must all use their own parameters. Every call of a burst
gives the bits of the same call made alone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcmod():
    from paper_2503_19379_gb300 import build as b
    b.build()
    import paper_2503_19379_gb300 as p
    return p


@pytest.mark.parametrize("lattice", [None, 0.5 * np.array([[0.0, 1.0, 1.0], [1.0, 0.0, 1.0], [1.0, 1.0, 0.0]])])
def test_burst_of_calls_keeps_each_calls_parameters(pcmod, lattice):
    N = 16
    g = np.random.default_rng(1)
    s = pcmod.Solver(N, g.uniform(1.0, 13.0, (3, N, N, N)), lattice=lattice)
    calls = []
    for i, nb in enumerate([3, 1, 7, 2, 12, 1, 5, 5]):
        k = g.uniform(-3.0, 3.0, (nb, 3))
        X = torch.randn(nb, 4, 3, N, N, N, dtype=torch.complex64 if i % 2 else torch.complex128, device="cuda")
        calls.append((s.apply_op if i % 3 else s.apply_precond, k, 2.0 * np.maximum(N, 1.0 / (k * k).sum(1)), X))
    burst = [f(k, gam, X) for f, k, gam, X in calls]
    torch.cuda.synchronize()
    for (f, k, gam, X), y in zip(calls, burst):
        alone = f(k, gam, X)
        torch.cuda.synchronize()
        assert torch.equal(y, alone)


def test_refused_under_capture(pcmod):
    """As before, a step call cannot be captured into a graph: it returns an error."""
    N = 8
    st = torch.cuda.Stream()
    s = pcmod.Solver(N, np.full((3, N, N, N), 2.0), stream=st.cuda_stream)
    X = torch.randn(1, 1, 3, N, N, N, dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with pytest.raises(Exception):
        with torch.cuda.graph(graph, stream=st):
            s.apply_op([[0.5, 0.2, 0.1]], [16.0], X)
    torch.cuda.synchronize()
