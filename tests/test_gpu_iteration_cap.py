"""The status of a solve at its iteration cap: a k-point that converges in the last iteration allowed has converged (plain
FP64 and mixed); one that needs another iteration has not (FP64) or is finished by the FP64 solve (mixed)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_converged_in_the_last_iteration(precision):
    from paper_2503_19379_gb300 import build as b
    b.build()
    import paper_2503_19379_gb300 as pcmod
    w = wl.workload_fcc_32()
    N, tol = 16, 1e-5
    eps = pcmod.eps_spheres(N, w.structure.as_array(), w.structure.eps_bg)

    def solve(maxiter):
        S = pcmod.Solver(N, eps, precision=precision, maxiter=maxiter)
        out = S.solve(w.kpts[[11]], 6, tol)
        S.close()
        return out

    n = int(solve(400)["iters"][0])
    seen = []
    for cap in range(max(1, n - 45) if precision else n - 1, n + 1):
        out = solve(cap)
        within = bool(np.all(out["resid"] <= tol))
        assert (out["status"] == 0) == within, (cap, out)
        seen.append((within, int(out["fp64_finish"][0])))
    assert (True, 0) in seen and ((False, 0) in seen or precision)
