"""The FP64 preconditioner forms two quotients per mode, 1 / (N^3 sigma) and ((gamma - 1) / gamma) / sigma, from one division.
The first is exact up to a power of two; the second is the product with the reciprocal, corrected by its remainder with two
fused multiply-adds, which rounds as the quotient itself does. Here in exact arithmetic (no GPU): the formula of the
z pass, and that the product alone does not (it rounds twice)."""
import os
import random
from fractions import Fraction as F

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_19379_gb300", "csrc")


def test_corrected_product_is_the_quotient():
    text = " ".join(open(os.path.join(CSRC, "fft.cu")).read().split())
    assert "f0 = fac * rs, f = fma(fma(-f0, sigma, fac), rs, f0)" in text
    rng = random.Random(5)
    rn = lambda x: F(float(x))  # float() of a fraction rounds to nearest, ties to even
    single = 0
    for _ in range(5000):
        gamma = rng.uniform(1.0, 600.0)
        fac, sigma = F((gamma - 1.0) / gamma), F(10.0 ** rng.uniform(-2.0, 6.0))
        rs = rn(1 / sigma)
        f0 = rn(fac * rs)
        f = rn(rn(fac - f0 * sigma) * rs + f0)
        assert f == rn(fac / sigma)
        single += f0 != f
    assert single > 500
