"""Complex128 Gram products: every entry is as accurate as FP64 products and sums make it, also where the columns are large in
different rows (an entry's products are then far smaller than the product of the columns' largest values).

Tolerance: the a-priori bound of FP64 sums of the 2 L real products, 2 L 2^-53 sum |a||b|, twice (the values of a span are
held to half a unit of 2^-53 of the largest, which is as much again), and 2^-1074 for each product that underflows.
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


def rand(g, *shape):
    return g.standard_normal(shape) + 1j * g.standard_normal(shape)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def check(got, A, B):
    ext = lambda x: x.astype(np.clongdouble)
    ref = np.einsum("bil,bjl->bij", ext(A.conj()), ext(B))
    size = np.einsum("bil,bjl->bij", np.abs(ext(A)), np.abs(ext(B)))
    err = np.abs(got - ref)
    tol = 4.0 * A.shape[2] * (2.0 ** -53 * size + np.longdouble(2.0) ** -1074)
    assert np.all(err <= tol), float(np.max(err / np.where(size == 0, 1, size)))


def panels(g, kind, nb, p, L):
    A = rand(g, nb, p, L)
    if kind == "spikes":  # each column has one value of 10^14 in a row where the others are zero
        for i in range(p):
            r = (7 * i + 3) % L
            A[:, :, r] = 0.0
            A[:, i, r] = 1e14 * (1 + 1j)
    elif kind == "apart":  # the columns' large parts do not overlap
        A *= 10.0 ** (-18.0 * ((np.arange(L)[None, :] * p // L) != np.arange(p)[:, None]))
    elif kind == "graded":  # every column falls off over 24 decades of rows, half of them the other way
        w = 10.0 ** (-24.0 * np.arange(L) / L)
        A[:, ::2] *= w
        A[:, 1::2] *= w[::-1]
    elif kind == "tiny":
        A[:, ::2] *= 2.0 ** -1000
        A[:, 1::2] *= 2.0 ** 400
    return A


@pytest.mark.parametrize("kind", ["dense", "spikes", "apart", "graded", "tiny"])
@pytest.mark.parametrize("nb,p,L", [(1, 3, 33), (2, 8, 1536), (1, 20, 1025), (1, 17, 3333), (1, 40, 640)])
def test_gram_pair_entries(pcmod, kind, nb, p, L):
    S = panels(np.random.default_rng(p), kind, nb, p, L)
    AS = S * np.random.default_rng(L).uniform(0.5, 4.0, L)
    G, H = (x.cpu().numpy() for x in pcmod.gram_pair(dev(S), dev(AS)))
    for got, B in ((G, S), (H, AS)):
        up = np.triu(got)
        check(up + np.triu(up, 1).conj().transpose(0, 2, 1), S, B)
        assert np.array_equal(got, got.conj().transpose(0, 2, 1))


@pytest.mark.parametrize("kind", ["dense", "spikes", "apart", "graded", "tiny"])
@pytest.mark.parametrize("nb,p,q,L", [(1, 1, 1, 5), (2, 9, 33, 700), (1, 64, 20, 2100), (1, 5, 48, 96)])
def test_gram_entries(pcmod, kind, nb, p, q, L):
    g = np.random.default_rng(q)
    A, B = panels(g, kind, nb, p, L), panels(g, kind, nb, q, L)
    check(pcmod.gram(dev(A), dev(B)).cpu().numpy(), A, B)
