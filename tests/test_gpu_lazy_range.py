"""Corrections that run without clamps first, and the level-0 value table's sums
by group, at the parameters where those forms are taken: a correction item is
lazy where S_0 <= limT (fast_fixed in items.cu), which the first test asserts for
parameters that saturate all the same; a level-0 thread adds up by group where
its samples times the largest squared value could leave 64 bits."""
import math

import numpy as np
import pytest

from paper_2502_07123_gb300 import workloads as W
from tests.test_gpu_chunk_forms import _parts, _same

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


def _lazy_limit(p, f, level, zmax):
    """limT 2^-f_S of a format with f_con1 >= f_mul1 >= f_sum1 and f_S >= f_mul2, or 0 where corrections keep
    their clamps: the bounds of fast_fixed.  zmax: the largest table value in units 2^-f_Z."""
    eS, (fZ, fc1, fc2, fm1, fs1, fm2, fS) = f["e"][6], f["f"]
    assert fc1 >= fm1 >= fs1 and fS >= fm2
    h = p["T"] / (1 << level)
    rnd = lambda x, b: math.floor(x * 2.0 ** b + 0.5)  # noqa: E731
    con1, con1c, con2 = rnd(p["r"] * h, fc1), rnd(p["r"] * 2 * h, fc1), rnd(p["sigma"] * math.sqrt(h), fc2)
    zc = 2 * zmax
    half = lambda k: 1 << (k - 1) if k > 0 else 0  # noqa: E731
    rs1, rs3, rss = fc2 + fZ - fm1, fc1 + 2 * fZ - fm1, fc1 - fs1
    mul = max((con2 * zc + half(rs1)) >> rs1, -((-con2 * zc + half(rs1)) >> rs1))
    if p["scheme"] == W.MILSTEIN:
        con3, one = rnd(0.5 * p["sigma"] ** 2 * h, fc1), 1 << 2 * fZ
        mul += max(abs((con3 * (zc * zc - one) + half(rs3)) >> rs3), abs((con3 * -2 * one + half(rs3)) >> rs3))
    spread = mul << (fc1 - fm1)
    sum1 = ((max(abs(con1), abs(con1c)) + half(rss) + spread) >> rss) + 1
    lim, mulS = (1 << (eS + fS)) - 1, 1 << (fS - fm2)
    add = (((lim * sum1 + half(fS + fs1 - fm2)) >> (fS + fs1 - fm2)) + 1) * mulS
    a, n = sum1 * 2.0 ** -fs1, 1 << level
    if lim + add >= 2 ** 31 - 1 or (min(con1, con1c) + half(rss) - spread) >> rss < -(1 << fs1):
        return 0.0
    if 2 * mulS * ((1 + a) ** n - 1) / a > lim:
        return 0.0
    return (((lim - mulS) << fs1) // ((1 << fs1) + sum1)) * 2.0 ** -fS


@pytest.mark.parametrize("payoff", [W.EURO, W.DIGITAL, W.ASIAN, W.LOOKBACK])
@pytest.mark.parametrize("scheme", [W.EULER, W.MILSTEIN])
@pytest.mark.parametrize("level,d,sigma,method", [(1, 3, 0.2, 1), (1, 4, 0.1, 1), (2, 3, 0.2, 1), (3, 4, 0.2, 1),
                                                  (5, 10, 0.2, 1), (6, 10, 0.2, 1), (4, 8, 0.2, 2)])
def test_lazy_corrections_that_saturate(m, payoff, scheme, level, d, sigma, method):
    """S limited to 128; S_0 just below limT; against the record-writing kernel, which clamps every step."""
    zs = np.abs(m.mlmc_icdf_method2_table(d, 2, 4, 12) if method == 2 else m.mlmc_icdf_table(1, d, 4, 12))
    zmax = int(round(float(zs.max()) * 2 ** 12))
    p = W.params(payoff=payoff, scheme=scheme, sigma=sigma, S0=60.0, K=60.0)
    fmts = [W.default_format(p, lev) for lev in range(level + 1)]
    for f in fmts:
        f["e"][6], f["e"][5] = 7, 7 + f["e"][4]
    lim_t = _lazy_limit(p, fmts[level], level, zmax)
    p["S0"] = p["K"] = math.floor(lim_t * 16 - 1) / 16
    assert 16 < p["S0"] <= lim_t
    P = m.make_params(p, d=d, method=method, formats=fmts)
    N = 60_011
    s = m.mlmc_level(level, N, P, m.NESTED_CORR_FIXED, 21, 4)
    t, rec = m.mlmc_level_dump(level, N, P, m.NESTED_CORR_FIXED, 21, 4)
    assert s["saturations"] == t["saturations"] == int(rec["sat"].sum()) and s["saturations"] > 20
    _same(s, t, N)


@pytest.mark.parametrize("pack", [0, 1])
def test_level0_sums_by_group(m, pack):
    """f_S = 21: 2^4 squared values of 30 bits fit 64 bits; a thread has more samples, in the parts it has 4 or 12."""
    p = W.params(payoff=W.EURO)
    f = W.default_format(p, 0)
    f["f"][6] = 21
    assert f["e"][6] + f["f"][6] == 30
    P = m.make_params(p, formats=[f], rng_pack=pack)
    N, per_group = 4_000_003, 12 if pack else 4
    info = m.Plan([dict(params=P, level=0, variant=m.FIXED_APPROX, N=N, first_sample=2)], 3).launch_info(0)
    assert N / (128 * info[2]) > 16
    s = m.mlmc_level(0, N, P, m.FIXED_APPROX, 3, 2)
    _same(s, _parts(m, 0, N, P, m.FIXED_APPROX, 3, 2, 128 * 512 // 12 * per_group), N)


@pytest.mark.parametrize("variant", ["FP16_APPROX", "BF16_APPROX", "FP16S_APPROX", "BF16S_APPROX"])
@pytest.mark.parametrize("payoff,scheme", [(W.EURO, W.EULER), (W.ASIAN, W.MILSTEIN), (W.LOOKBACK, W.EULER)])
def test_two_deep_samples_per_thread(m, variant, payoff, scheme):
    """Level 8: a thread has two samples from 24 chunks per SM on; the parts give it one."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    P = m.make_params(W.params(payoff=payoff, scheme=scheme))
    N = 2 * 128 * 24 * sms + 131
    info = m.Plan([dict(params=P, level=8, variant=getattr(m, variant), N=N, first_sample=11)], 7).launch_info(0)
    assert info[2] == -(-N // 256)
    s = m.mlmc_level(8, N, P, getattr(m, variant), 7, 11)
    _same(s, _parts(m, 8, N, P, getattr(m, variant), 7, 11, 70_001), N)
