"""The FP64 exact kernels against the oracle where their datapath changes: the
integer increments' range (sigma sqrt(h) up to about 0.6 on one step, half that
with a coarse path) and the FP64 increments beyond it, zero and negative
constants, every payoff class and scheme."""
import numpy as np
import pytest

from oracle import core
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


@pytest.mark.parametrize("payoff", [W.EURO, W.DIGITAL, W.ASIAN, W.LOOKBACK])
@pytest.mark.parametrize("scheme", [W.EULER, W.MILSTEIN])
@pytest.mark.parametrize("level,sigma,r", [(0, 0.6, 0.05), (0, 1.5, 0.05), (1, 0.8, 0.05), (1, 2.0, -0.3),
                                           (3, 0.0, 0.0), (3, 0.3, -0.4), (4, 3.0, 0.0), (8, 0.2, 0.05)])
def test_datapaths(m, payoff, scheme, level, sigma, r):
    """Terminal values to 1e-12 of the largest of |S| and S0 (a step's rounding is a
    few 2^-53 of either); payoffs to four times that of the path scale."""
    p = W.params(payoff=payoff, scheme=scheme, sigma=sigma, r=r)
    first, N, seed = 5, 203, 91 + level
    _, g = m.mlmc_level_dump(level, N, m.make_params(p, request=2), m.FP64_EXACT, seed, first)
    s = m.mlmc_level(level, N, m.make_params(p, request=2), m.FP64_EXACT, seed, first)
    _, o = core.level(p, level, first, N, core.FP64_EXACT, seed, request=2, dump=True)
    scale = np.maximum(np.abs(o["sf"]), p["S0"]) + np.abs(o["sc"])
    if sigma >= 1.5 and level > 0:   # such paths change sign on the way: their running maximum bounds them
        scale = scale * (1.0 + 6.4 * sigma * 2.0 ** (-level / 2)) ** 4
    for f in ("sf", "sc"):
        assert np.all(np.abs(g[f] - o[f]) <= 1e-12 * scale), f
    for f, t in (("pf", "sf"), ("pc", "sc")):
        near = np.abs(o[t] - p["K"]) <= 4e-12 * scale if payoff == W.DIGITAL else False
        assert np.all((np.abs(g[f] - o[f]) <= 4e-12 * scale) | near), f
    disc = np.exp(-p["r"] * p["T"])
    assert abs(s["sum"] - disc * g["y"].sum()) <= 1e-12 * disc * np.abs(g["y"]).sum() + 1e-300
