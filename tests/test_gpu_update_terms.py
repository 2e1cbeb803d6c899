"""Complex128 block updates: every output is as accurate as its own terms, however small they are beside the others of the
row (columns of very different sizes, a C that picks or scales single columns).

Tolerance. An output formed from digits has a term within 2^G of the largest product of its row, 2^G sqrt(2 p) <= 2^6.2, and
an error of 2^-60.2 sqrt(2 p) (rms) of that product: 2^-54 of sum |s||c|, 2^-51.4 at six standard deviations, and one
rounding. The others are FP64 sums of 2 p products: 2^-54.8 (rms) of at most sum |s||c| for each rounding, 2^-52.2 sqrt(2 p)
at six standard deviations. Outputs of a single product need two roundings, 2^-52.
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


def error_of_terms(pcmod, S, C):
    """The largest error of an output over the sum of its terms' magnitudes."""
    Y = pcmod.block_update(dev(S), dev(C)).cpu().numpy()
    ext = lambda A: A.astype(np.clongdouble)
    ref = np.einsum("bpl,bpq->bql", ext(S), ext(C))
    size = np.einsum("bpl,bpq->bql", np.abs(ext(S)), np.abs(ext(C)))
    err = np.abs(Y - ref)
    assert np.all(err[size == 0] == 0)
    return float(np.max(err / np.where(size == 0, 1, size)))


# graded: columns 1, 10^-d, 10^-2d, ...; C: identity, diagonal over 10^-12..10^12, two blocks
@pytest.mark.parametrize("p,L", [(2, 300), (13, 129), (33, 260), (48, 1000), (64, 500)])
@pytest.mark.parametrize("kind", ["identity", "diagonal", "blocks"])
def test_graded_columns_keep_their_digits(pcmod, p, L, kind):
    g = np.random.default_rng(p)
    q = min(p, 24)
    S = rand(g, 2, p, L) * 10.0 ** (-20.0 * np.arange(p) / max(p - 1, 1))[:, None]
    C = np.zeros((2, p, q), dtype=np.complex128)
    if kind == "blocks":
        h, r = p // 2, q // 2
        C[:, :h, :r], C[:, h:, r:] = rand(g, 2, h, r), rand(g, 2, p - h, q - r)
    else:
        C[:, np.arange(q), np.arange(q)] = 1.0 if kind == "identity" else 10.0 ** g.uniform(-12, 12, (2, q))
    tol = 2.0 ** -51 + 2.0 ** -52.2 * np.sqrt(2 * p) if kind == "blocks" else 2.0 ** -52
    assert error_of_terms(pcmod, S, C) <= tol


@pytest.mark.parametrize("p,q,L", [(1, 1, 64), (3, 3, 200), (8, 4, 1536), (17, 17, 300), (48, 16, 2000), (64, 33, 700)])
def test_near_identity_and_dense_coefficients(pcmod, p, q, L):
    """A rotation close to the identity leaves outputs whose largest term is small where their column is; dense random
    coefficients leave none."""
    g = np.random.default_rng(q + p)
    S = rand(g, 2, p, L)
    C = 1e-7 * rand(g, 2, p, q)
    C[0, np.arange(q), np.arange(q)] += 1.0
    tol = 2.0 ** -51 + 2.0 ** -52.2 * np.sqrt(2 * p)
    assert error_of_terms(pcmod, S, C) <= tol


def test_scales_far_from_one(pcmod):
    """Entries of 2^-1000 against coefficients of 2^900, zero rows, columns and coefficients."""
    g = np.random.default_rng(5)
    S, C = rand(g, 1, 20, 400), rand(g, 1, 20, 9)
    S[0, 3] *= 2.0 ** -1000
    C[0, 3] *= 2.0 ** 900
    S[0, 5], C[0, 6], C[0, :, 4], S[0, :, 77] = 0.0, 0.0, 0.0, 0.0
    C[0, :3, 7] = C[0, 4:, 7] = 0.0  # output 7: only the scaled column
    assert error_of_terms(pcmod, S, C) <= 2.0 ** -51 + 2.0 ** -52.2 * np.sqrt(40)


@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
def test_sum_of_no_columns(pcmod, dtype):
    """p = 0 through the C ABI: zeros in the outputs, nothing past them."""
    from paper_2503_19379_gb300 import pc
    Y = torch.ones(3, 5, 37, dtype=dtype, device="cuda")
    z = torch.zeros(1, dtype=torch.complex128, device="cuda")
    rc = pcmod.lib().pc_block_update(3, 37, 0, 4, pc._dtype_code(Y), pc._dev(z), 0, pc._dev(z), pc._dev(Y), 5 * 37,
                                     pc._stream(None))
    assert rc == 0
    assert bool((Y[:, :4] == 0).all()) and bool((Y[:, 4] == 1).all())
