"""The warm start's forward pass and gradient with a predicted block X that is aligned to one complex64 (8 bytes) only: the same
block bit for bit as in an aligned buffer, and the gradient of the aligned one within the rounding of its FP32 sums (other
kernels for panels that are not 16-byte aligned: 1e-4 of the largest entry)."""
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


@pytest.mark.parametrize("N,nb,S", [(16, 3, 2), (32, 8, 3), (16, 10, 2), (16, 16, 2)])
def test_x_offset_by_one_element(pcmod, N, nb, S):
    from paper_2503_19379_gb300 import pc
    g = np.random.default_rng(N)
    net = pcmod.WarmStart(N, nb, S)
    net.params.copy_(torch.from_numpy(0.3 * g.standard_normal(net.P).astype(np.float32)))
    m0 = torch.from_numpy(g.uniform(0.1, 1.0, (2, 3, N, N, N)).astype(np.float32)).cuda()
    sidx = torch.tensor([i % 2 for i in range(S)], dtype=torch.int32, device="cuda")
    k = np.ascontiguousarray(g.uniform(-3, 3, (S, 3)))
    gen = torch.Generator(device="cuda").manual_seed(N)
    V = torch.randn(S, nb, 3, N, N, N, dtype=torch.complex64, device="cuda", generator=gen) / np.sqrt(3 * N ** 3)
    lam = torch.from_numpy(np.sort(g.uniform(2.0, 60.0, (S, nb)), axis=1)).cuda()
    X, y = net.forward(m0, sidx, k)
    grad, loss = net.backward(m0, sidx, X, y, V, lam)
    buf = torch.zeros(X.numel() + 2, dtype=torch.complex64, device="cuda")
    X1 = buf[1:-1].view(X.shape)
    assert X1.data_ptr() % 16 == 8
    y1 = torch.empty_like(y)
    rc = pcmod.lib().pc_ws_forward(N, nb, S, pc._dev(net.params), pc._dev(m0), 2, pc._dev(sidx), pc._dptr(k), pc._dev(X1),
                                   pc._dev(y1), pc._dev(net.work), pc._stream(None))
    assert rc == 0 and torch.equal(X1, X) and torch.equal(y1, y)
    assert complex(buf[0]) == 0 and complex(buf[-1]) == 0
    grad1, loss1 = net.backward(m0, sidx, X1, y1, V, lam)
    assert float((grad1 - grad).abs().max()) <= 1e-4 * float(grad.abs().max())
    assert float((loss1 - loss).abs().max()) <= 1e-5 * nb
