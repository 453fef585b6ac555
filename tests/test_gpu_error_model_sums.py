"""The error model's sums of many nearly equal terms.  On level 0 S_1 / (1 + sum1_0)
is S_0, so every sample in the money adds (e^-rT S_0)^2 to the mul1 and con1
instances up to its own roundings, which average out over the samples, while
the roundings of sums of like terms do not."""
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_2502_07123_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2502_07123_gb300 import mlmc
    return mlmc


@pytest.mark.parametrize("sigma", [0.1, 0.2, 0.4])
@pytest.mark.parametrize("N", [20_000, 400_001, 4_000_003])
def test_like_terms(m, N, sigma):
    """At most one rounding (2^-53) for each of the 7 foldings of a CTA's 128 samples, the 7 steps that
    join 128 columns of CTAs, the division by N and the constant, and 1/2 for the terms' mean."""
    p = W.params(sigma=sigma)
    g = m.mlmc_sensitivities(0, N, m.make_params(p), 17, 3, per_instance=True)
    d = m.mlmc_level(0, N, m.make_params(W.params(sigma=sigma, payoff=W.DIGITAL)), m.FP64_EXACT, 17, 3)
    disc = math.exp(-p["r"] * p["T"])
    inside = round(d["sum"] / disc)
    want = (Fraction(disc) * Fraction(p["S0"])) ** 2 * inside / N
    inst = np.asarray(g["inst"]).reshape(7, -1)
    for t in (3, 1):   # mul1 and con1, fine step 0
        assert abs(Fraction(float(inst[t][0])) / want - 1) <= Fraction(33, 2) / 2 ** 53, t
