"""A wait that runs out inside a tensor-core kernel leaves garbage, so the calls that run these kernels look for it once
they have synchronised: the Gram products, the plain FP64 solve, the mixed solve. The time-out is put into the word that the
kernels report to, on the host; the kernels themselves run as always. The call that finds it fails, and the next does not."""
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


def calls(pcmod):
    gen = torch.Generator(device="cuda").manual_seed(1)
    S = torch.randn(1, 20, 1536, dtype=torch.complex128, device="cuda", generator=gen)
    F = S.to(torch.complex64)
    yield "gram", lambda: pcmod.gram(S, S)
    yield "gram_pair", lambda: pcmod.gram_pair(S, S)
    yield "gram c64", lambda: pcmod.gram(F, F)
    yield "gram_pair_coupled", lambda: pcmod.gram_pair_coupled(F, F, F[:, :4].contiguous())
    eps = pcmod.eps_spheres(8, [[0.5, 0.5, 0.5, 0.3, 13.0]], 1.0)
    for precision in (0, 1):
        for kchunk in (0, 1):
            s = pcmod.Solver(8, eps, precision=precision, kchunk=kchunk)
            yield f"solve {precision} {kchunk}", lambda: s.solve([[0.9, 0.4, -0.3], [1.7, -0.2, 0.8]], 4, 1e-6)


def test_a_timeout_is_reported_once(pcmod):
    L = pcmod.lib()
    for name, call in calls(pcmod):
        call()
        L.pc_inject_tc_timeout(1)
        with pytest.raises(pcmod.PCError, match="ran out of time"):
            call()
            pytest.fail(name)
        out = call()
        if name.startswith("solve"):
            assert out["status"] == 0 and np.all(out["resid"] <= 1e-6)


def test_the_fp64_finish_looks_too(pcmod):
    eps = pcmod.eps_spheres(16, [[0.5, 0.5, 0.5, 0.3, 13.0]], 1.0)
    k = [[0.9, 0.4, -0.3]]
    s = pcmod.Solver(16, eps, precision=1, maxiter=8)  # (it needs about 20)
    ref = s.solve(k, 4, 1e-6)
    assert ref["fp64_finish"][0] == 1
    pcmod.lib().pc_inject_tc_timeout(2)
    with pytest.raises(pcmod.PCError, match="ran out of time"):
        s.solve(k, 4, 1e-6)
    out = s.solve(k, 4, 1e-6)
    assert out["status"] == ref["status"] and np.allclose(out["evals"], ref["evals"], rtol=1e-6, atol=0.0)
