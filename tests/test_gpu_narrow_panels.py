"""Complex64 panels through the C ABI at the widths and lengths where their CUDA-core kernels change form: narrow Gram
products (p, q <= 16, tiles of 8 x 8 outputs) and block updates large enough for two rows a thread (even lengths,
16-byte aligned).

Tolerances. Gram: FP32 sums of a few dozen products a thread and over a warp's lanes, FP64 above that: 4e-6 of
|A|^H |B|, as for the other complex64 products. Update: FP32 products and sums of 2 p terms, 8 eps32 sqrt(p) of
max |S| max |C| with a factor 2 for the two parts.
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
    return g.standard_normal(shape) + 1j * g.standard_normal(shape)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("nb,p,q,L", [(1, 1, 1, 1), (2, 8, 8, 127), (3, 9, 16, 129), (1, 16, 9, 4097), (16, 8, 8, 12288),
                                      (2, 16, 16, 98304), (1, 4, 5, 512), (300, 3, 12, 600)])
def test_gram_narrow_c64(pcmod, nb, p, q, L):
    A, B = rand(p, (nb, p, L)).astype(np.complex64), rand(q + 50, (nb, q, L)).astype(np.complex64)
    G = pcmod.gram(dev(A), dev(B)).cpu().numpy()
    A, B = A.astype(np.complex128), B.astype(np.complex128)
    bound = (np.abs(A.real) + np.abs(A.imag)) @ (np.abs(B.real) + np.abs(B.imag)).transpose(0, 2, 1)
    assert np.all(np.abs(G - A.conj() @ B.transpose(0, 2, 1)) <= 4e-6 * bound)


@pytest.mark.parametrize("nb,p,q,L", [(2, 38, 8, 90002), (1, 1, 1, 160000), (2, 64, 9, 90002), (2, 57, 19, 90002),
                                      (1, 17, 33, 90002), (3, 33, 24, 60006), (2, 12, 16, 90002), (2, 20, 12, 90003)])
def test_block_update_two_rows(pcmod, nb, p, q, L):
    S = rand(p, (nb, p, L)).astype(np.complex64)
    C = rand(q, (nb, p, q))
    Y = pcmod.block_update(dev(S), dev(C)).cpu().numpy()
    ref = C.transpose(0, 2, 1) @ S.astype(np.complex128)
    bound = 16 * np.finfo(np.float32).eps * np.sqrt(p) * np.max(np.abs(S)) * np.max(np.abs(C))
    assert np.max(np.abs(Y - ref)) <= bound
