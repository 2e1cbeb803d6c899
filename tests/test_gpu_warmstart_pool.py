"""The warm start's channel means: a network whose features are one constant (zero convolution weights) gives y = that
constant, summed over (N/4)^3 points.

Tolerance: 256 sums of (N/4)^3 / 256 terms in FP32, then eight levels. Each addition rounds by at most 2^-24 of a partial sum,
half the total on average: ((N/4)^3 / 512 + 8) 2^-24, and four roundings of the products around it."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcmod():
    from paper_2503_19379_gb300 import build as b
    b.build()
    import paper_2503_19379_gb300 as p
    return p


@pytest.mark.parametrize("N", [16, 32, 64, 128, 256])
@pytest.mark.parametrize("value", [1.1, 1.3, 0.7])
def test_mean_of_a_constant(pcmod, N, value):
    net = pcmod.WarmStart(N, 1, 1)
    sizes = [8 * 81, 8, 16 * 216, 16, 96, 16, 96, 16, 6 * 16, 6, 22, 1]
    at = [sum(sizes[:i]) for i in range(len(sizes))]
    net.params.zero_()
    net.params[at[3]:at[3] + 16] = value  # b2: the features of every channel
    net.params[at[10]] = 1.0  # Wv: channel 0
    _, y = net.forward(torch.ones(1, 3, N, N, N, dtype=torch.float32, device="cuda"),
                       torch.zeros(1, dtype=torch.int32, device="cuda"), [[0.3, 0.2, 0.1]])
    ref = float(torch.tensor(value, dtype=torch.float32))
    assert abs(float(y[0, 0]) - ref) <= (((N // 4) ** 3 / 512 + 8) + 4) * 2.0 ** -24 * ref
