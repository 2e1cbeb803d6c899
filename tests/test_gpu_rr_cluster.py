"""The Rayleigh-Ritz kernel divides a pencil over 4, 2 or 1 thread blocks, by the batch size. No entry's arithmetic depends
on the division, so the same pencil gives the same bits in batches of every size, at full and at reduced rank."""
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


@pytest.mark.parametrize("n,m,rank", [(1, 1, 1), (3, 2, 3), (5, 5, 5), (24, 8, 24), (39, 13, 20), (57, 19, 57), (64, 21, 64),
                                      (64, 64, 64), (12, 6, 3)])
def test_same_bits_for_every_cluster_size(pcmod, n, m, rank):
    g = np.random.default_rng(100 * n + m)
    S = g.standard_normal((200, rank)) + 1j * g.standard_normal((200, rank))
    S = S @ (g.standard_normal((rank, n)) + 1j * g.standard_normal((rank, n)) if rank < n else np.eye(n))
    G, H = S.conj().T @ S, S.conj().T @ (np.linspace(1.0, 50.0, 200)[:, None] * S)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    out = []
    for nb in (1, sms // 4 + 1, sms // 2 + 1):  # 4, 2 and 1 blocks per pencil
        Gt, Ht = (torch.from_numpy(np.tile(x, (nb, 1, 1))).cuda() for x in (G, H))
        theta, coef, rk = pcmod.rayleigh_ritz(Gt, Ht, m, 1e-12)
        assert torch.equal(theta, theta[:1].expand_as(theta)) and torch.equal(coef, coef[:1].expand_as(coef))
        out.append((theta[0], coef[0], int(rk[0])))
    for theta, coef, rk in out[1:]:
        assert rk == out[0][2] == min(n, rank)
        assert torch.equal(theta, out[0][0]) and torch.equal(coef, out[0][1])
