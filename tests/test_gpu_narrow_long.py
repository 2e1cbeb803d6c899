"""Narrow complex64 Gram products (p, q <= 16) of long panels in large batches, where a thread's share of the rows is
hundreds of rows: constant columns, whose products all round the same way, so that a long FP32 sum drifts.

Tolerance: at most 64 rows a thread are summed in FP32 before they go to FP64 (128 products, five levels over the lanes).
Each of the 133 additions rounds by at most 2^-24 of a partial sum, which is half the total on average: 4e-6.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcmod():
    from paper_2503_19379_gb300 import build as b
    b.build()
    import paper_2503_19379_gb300 as p
    return p


@pytest.mark.parametrize("nb,p,L", [(1300, 2, 98304), (64, 4, 786432), (1, 9, 64), (3, 16, 8193)])
def test_long_narrow_panels(pcmod, nb, p, L):
    v = torch.tensor([1.1 + 0.3j, 1.3 + 0.7j, 0.9 + 1.01j, 3.1], dtype=torch.complex64, device="cuda")[torch.arange(p) % 4]
    A = v[None, :, None].expand(nb, p, L).contiguous()
    w = v.to(torch.complex128)
    ref = L * w.conj()[:, None] * w[None, :]
    size = L * (w.real.abs() + w.imag.abs())[:, None] * (w.real.abs() + w.imag.abs())[None, :]
    G = pcmod.gram(A, A)
    assert float(((G - ref).abs() / size).max()) <= 4e-6
