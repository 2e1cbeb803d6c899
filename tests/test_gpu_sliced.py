"""Products of FP64-accurate panels on the tensor cores (exact FP16 digit slices) through the C ABI.

Tolerance of the Gram products. A value is rounded to an integer m whose largest in the column is at least 2^53 (M): a
uniform error of +-1/2, rms 2^-54.8 M, and 2^-54.3 M_a M_b for each of the 2 L real products of an entry; the digit
pairs of levels 8 and above are far smaller. Six standard deviations of their sum, 6 sqrt(2 L) 2^-54.2 M_a M_b, bound it;
the FP64 sums over spans and chunks add a few 2^-53 of the entry.

Block updates: one exponent per row and per column of the coefficients (scaled by the largest entry of their row), eight
digits (m up to 2^61 and more): T = max_i(|s_li| c_i) max_i(|c_ij| / c_i) takes the place of M_a M_b. The seven digit
pairs of level 8 are dropped, 2^(48 + 12.4 + 1.4) of 2^122 (random digits, rms 74 each): 2^-60.2 T (rms) for each of
the 2 p real products, and the total is rounded once.
"""
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


def rand(seed, shape):
    g = np.random.default_rng(seed)
    x = g.standard_normal(shape) + 1j * g.standard_normal(shape)
    return x * np.exp(2.0 * g.standard_normal(shape[:-1]))[..., None]  # columns of different sizes


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def top(A):
    return np.maximum(np.abs(A.real), np.abs(A.imag)).max(axis=2)


def check(got, A, B, upper=False):
    L = A.shape[2]
    # the reference sums in extended precision, so that its own rounding stays below the tolerance
    ref = np.einsum("bil,bjl->bij", A.conj().astype(np.clongdouble), B.astype(np.clongdouble))
    tol = 6.0 * np.sqrt(2.0 * L) * 2.0 ** -54.2 * top(A)[:, :, None] * top(B)[:, None, :] + 2.0 ** -50 * np.abs(ref)
    ratio = np.abs(got - ref) / np.maximum(tol, np.finfo(np.float64).tiny)
    if upper:
        ratio = np.triu(ratio)
    assert np.all(ratio <= 1.0), float(np.max(ratio))


@pytest.mark.parametrize("nb,p,L", [(1, 1, 1), (2, 16, 31), (1, 17, 33), (3, 32, 128), (1, 33, 129), (2, 48, 1025),
                                    (1, 64, 2100), (4, 21, 1536), (1, 39, 12288)])
def test_gram_pair_sliced(pcmod, nb, p, L):
    S = rand(p + L, (nb, p, L))
    w = np.random.default_rng(L).uniform(0.5, 40.0, L)
    AS = S * w
    G, H = (x.cpu().numpy() for x in pcmod.gram_pair(dev(S), dev(AS)))
    for got, B in ((G, S), (H, AS)):
        check(got, S, B, upper=True)  # the lower triangle is its mirror
        assert np.array_equal(got, got.conj().transpose(0, 2, 1))


@pytest.mark.parametrize("nb,p,q,L", [(1, 1, 1, 7), (2, 5, 33, 640), (1, 64, 64, 1500), (3, 40, 32, 96),
                                      (1, 12, 24, 999)])
def test_gram_sliced(pcmod, nb, p, q, L):
    A, B = rand(p, (nb, p, L)), rand(100 + q, (nb, q, L))
    check(pcmod.gram(dev(A), dev(B)).cpu().numpy(), A, B)


@pytest.mark.parametrize("bits", [0x3FFFFFFFFFFFFFFF, 0x3FF7F7F7F7F7F7F7, 0x3FF8080808080808])
def test_gram_extreme_digits(pcmod, bits):
    """Constant columns whose digits are all at an end of their range: the level sums are the largest possible, and a
    rounding of the accumulator would show. All products are equal, so only the dropped levels' part remains:
    at most 5 2^46 of 2^106 per product, below the rounding of the FP64 sums over spans."""
    v = np.array([bits], dtype=np.uint64).view(np.float64)[0]
    L = 4096
    S = np.full((1, 64, L), v * (1 - 1j))
    G, _ = (x.cpu().numpy() for x in pcmod.gram_pair(dev(S), dev(S)))
    ref = float(2 * np.longdouble(v) ** 2 * L)
    assert np.max(np.abs(G - ref)) <= 8 * 2.0 ** -53 * ref


def test_gram_nonfinite(pcmod):
    """An infinity or a NaN reaches exactly the entries of its columns, as in plain FP64 sums."""
    S = rand(3, (1, 10, 2500))
    S[0, 3, 1500] = np.inf
    S[0, 7, 10] = np.nan
    G, H = (x.cpu().numpy()[0] for x in pcmod.gram_pair(dev(S), dev(S)))
    touched = np.zeros((10, 10), dtype=bool)
    touched[[3, 7], :] = touched[:, [3, 7]] = True
    assert np.array_equal(~np.isfinite(G.real), touched) and np.array_equal(~np.isfinite(H.real), touched)
    ok = [i for i in range(10) if i not in (3, 7)]
    check(G[None][:, ok][:, :, ok], S[:, ok], S[:, ok])


def test_gram_zero_and_tiny_columns(pcmod):
    """Zero columns give exact zeros; a column of a scale far from the others' keeps its relative accuracy."""
    S = rand(4, (1, 6, 700))
    S[0, 2] = 0.0
    S[0, 4] *= 2.0 ** -300
    S[0, 5] *= 2.0 ** 300
    G, _ = (x.cpu().numpy() for x in pcmod.gram_pair(dev(S), dev(S)))
    assert np.all(G[0, 2] == 0.0) and np.all(G[0, :, 2] == 0.0)
    check(G, S, S)


def check_update(Y, S, C):
    p = S.shape[1]
    ref = np.einsum("bpl,bpq->bql", S.astype(np.clongdouble), C.astype(np.clongdouble))
    part = lambda A: np.maximum(np.abs(A.real), np.abs(A.imag))
    ci = part(C).max(axis=2)
    T = (part(S) * ci[:, :, None]).max(axis=1)[:, None, :] * (part(C) / ci[:, :, None]).max(axis=1)[:, :, None]
    tol = 6.0 * np.sqrt(2.0 * p) * 2.0 ** -59.5 * T + 2.0 ** -52 * np.abs(ref)
    ratio = np.abs(Y - ref) / tol
    assert np.all(ratio <= 1.0), float(np.max(ratio))


@pytest.mark.parametrize("nb,p,q,L", [(1, 1, 1, 1), (2, 16, 3, 127), (1, 17, 8, 129), (3, 32, 33, 640), (1, 33, 24, 1000),
                                      (2, 48, 25, 2500), (1, 49, 16, 128), (1, 64, 64, 5000), (200, 9, 4, 300)])
def test_block_update_sliced(pcmod, nb, p, q, L):
    S = rand(p + L, (nb, p, L))
    g = np.random.default_rng(q)
    C = g.standard_normal((nb, p, q)) + 1j * g.standard_normal((nb, p, q))
    C /= np.abs(S).max(axis=2)[:, :, None]  # small columns with large coefficients, as preconditioned residuals have
    check_update(pcmod.block_update(dev(S), dev(C)).cpu().numpy(), S, C)


def test_block_update_nonfinite_and_zero(pcmod):
    """An infinity stays in its row, a NaN coefficient in its column; zero rows give zeros."""
    S = rand(8, (1, 20, 400))
    g = np.random.default_rng(9)
    C = g.standard_normal((1, 20, 12)) + 1j * g.standard_normal((1, 20, 12))
    S[0, 4, 77] = np.inf
    S[0, :, 200] = 0.0
    Y = pcmod.block_update(dev(S), dev(C)).cpu().numpy()
    bad = ~np.isfinite(Y[0])
    assert bad[:, 77].all() and bad.sum() == 12 and np.all(Y[0, :, 200] == 0.0)
    S[0, 4, 77] = 1.0
    C[0, 3, 5] = np.nan
    Y = pcmod.block_update(dev(S), dev(C)).cpu().numpy()
    assert np.isnan(Y[0, 5]).all() and np.isfinite(np.delete(Y[0], 5, axis=0)).all()
    ok = [j for j in range(12) if j != 5]
    ref = np.einsum("pl,pq->ql", S[0], C[0][:, ok])
    assert np.max(np.abs(Y[0][ok] - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("nbands,guard", [(1, 0), (3, 1), (10, 6), (11, 6), (12, 9)])
def test_mixed_solve_block_widths(pcmod, nbands, guard):
    """The mixed solve's block X (double-float pairs: Gram and update) at 1, 4, 16, 17 and 21 columns. Residuals of
    1e-6 leave eigenvalue errors of about 1e-12 over the relative gap (at least 1e-4 here)."""
    N, k = 8, [[0.9, 0.4, -0.3], [1.7, -0.2, 0.8], [0.3, 2.1, 1.0]]
    eps = pcmod.eps_spheres(N, [[0.5, 0.5, 0.5, 0.3, 13.0]], 1.0)
    a = pcmod.Solver(N, eps, precision=1, guard=guard).solve(k, nbands, 1e-6)
    b = pcmod.Solver(N, eps, precision=0, guard=guard).solve(k, nbands, 1e-8)
    assert a["status"] == 0 and b["status"] == 0
    assert np.max(np.abs(a["evals"] - b["evals"]) / b["evals"]) <= 1e-8
