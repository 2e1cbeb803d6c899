"""The complex64 FFT preconditioner on a general cell at every split of the line transforms (N = 8, 16: one DFT; 32, 64,
128: a second DFT of length 2, 4, 8 in the middle steps), against the oracle's FFT solve in FP64: 2e-5 of the largest entry,
the tolerance of the cube's complex64 preconditioner."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from oracle import precond  # noqa: E402

pytestmark = pytest.mark.gpu

CELL = np.array([[1.0, 0.3, -0.2], [0.1, 0.9, 0.25], [-0.15, 0.2, 1.1]])


@pytest.fixture(scope="module")
def pcmod():
    from paper_2503_19379_gb300 import build as b
    b.build()
    import paper_2503_19379_gb300 as p
    return p


@pytest.mark.parametrize("N,nb,m,variant", [(8, 3, 2, 0), (16, 1, 3, 0), (32, 2, 2, 0), (32, 1, 1, 1), (64, 2, 1, 0),
                                            (128, 1, 1, 0)])
def test_precond_c64_lattice_sizes(pcmod, N, nb, m, variant):
    S = pcmod.Solver(N, np.ones((3, N, N, N)), lattice=CELL, precond=variant)
    g = np.random.default_rng(N + variant)
    kpts = g.uniform(-3, 3, (nb, 3))
    kpts[-1] *= nb == 1  # the last of several is k = 0
    gammas = np.linspace(2.0 * N, 5.0 * N, nb)
    R = (g.standard_normal((nb, m, 3 * N ** 3)) + 1j * g.standard_normal((nb, m, 3 * N ** 3))).astype(np.complex64)
    W = S.apply_precond(kpts, gammas, torch.from_numpy(R.reshape(nb, m, 3, N, N, N)).cuda()).cpu().numpy()
    for b in range(nb):
        for j in range(m):
            ref = precond.apply_preconditioner(R[b, j].astype(np.complex128), N, 1.0 / N, kpts[b], gammas[b], 1,
                                               "laplacian" if variant else "gamma", CELL).ravel()
            assert np.max(np.abs(W[b, j].ravel() - ref)) <= 2e-5 * np.max(np.abs(ref))
