"""The pinned staging of contexts comes from a pool of returned blocks: contexts made one after the other allocate no more of
it than one of them, and contexts made, used and closed by several threads at once each get blocks of their own."""
import threading

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


def test_contexts_in_turn_reuse_the_blocks(pcmod):
    count = pcmod.lib().pc_pinned_allocations
    eps = np.full((3, 8, 8, 8), 2.0)
    pcmod.Solver(8, eps).close()
    before = count()
    for _ in range(10):
        pcmod.Solver(8, eps).close()
    assert count() == before


def test_threads_get_blocks_of_their_own(pcmod):
    N, g = 8, np.random.default_rng(2)
    eps = g.uniform(1.0, 13.0, (3, N, N, N))
    X = torch.from_numpy(g.standard_normal((1, 2, 3, N, N, N)) + 1j * g.standard_normal((1, 2, 3, N, N, N))).cuda()
    kpts = g.uniform(-3.0, 3.0, (4, 12, 1, 3))
    torch.cuda.synchronize()
    got = [[None] * 12 for _ in range(4)]
    fails = []

    def work(t):
        try:
            for i in range(12):
                s = pcmod.Solver(N, eps)
                ys = [s.apply_op(kpts[t, i], [16.0], X) for _ in range(3)]  # more calls than staging slots
                torch.cuda.synchronize()
                assert torch.equal(ys[0], ys[2])
                got[t][i] = ys[1].cpu()
                s.close()
        except Exception as e:  # noqa: BLE001 (handed to the main thread)
            fails.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not fails, fails
    s = pcmod.Solver(N, eps)
    for t in range(4):
        for i in range(12):
            assert torch.equal(got[t][i], s.apply_op(kpts[t, i], [16.0], X).cpu())
