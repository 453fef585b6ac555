"""Chunked sums against the same samples summed otherwise, where the chunking or
the form of a chunk changes: the final sum of a few and of many chunks, larger
chunks of large items, two half-precision samples per thread, the level-0 value
table's two ways of summing, corrections that leave the lazy range, and the
error model's batches of 128 samples.  Integer sums are equal; real ones agree to
1e-12 of sum |Y| (the bound of the float pairs, 3.5e-13 on either side)."""
import math

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


def _parts(m, level, N, P, variant, seed, first, size):
    """mlmc_level over consecutive ranges of at most `size` samples, added up."""
    out = dict(isum=0, isum2=0, saturations=0, sum=0.0, sum2=0.0)
    for at in range(0, N, size):
        s = m.mlmc_level(level, min(size, N - at), P, variant, seed, first + at)
        for k in out:
            out[k] += s[k]
    return out


def _same(s, t, n):
    assert s["saturations"] == t["saturations"]
    if s["exact_int"]:
        assert (s["isum"], s["isum2"]) == (t["isum"], t["isum2"])
    else:   # sum |Y| <= sqrt(n sum Y^2)
        assert abs(s["sum"] - t["sum"]) <= 1e-12 * math.sqrt(n * t["sum2"])
        assert abs(s["sum2"] - t["sum2"]) <= 1e-12 * t["sum2"]


@pytest.mark.parametrize("chunks", [1, 31, 32, 33, 128, 129, 500])
@pytest.mark.parametrize("variant", ["FIXED_APPROX", "FP32_EXACT", "FP64_EXACT", "NESTED_CORR_FIXED"])
def test_final_sum(m, variant, chunks):
    """128 samples per chunk; the parts have at most 8 chunks."""
    P = m.make_params(W.params(), request=1)
    N = 128 * chunks - 5
    s = m.mlmc_level(3, N, P, getattr(m, variant), 5, 3)
    _same(s, _parts(m, 3, N, P, getattr(m, variant), 5, 3, 1024), N)


@pytest.mark.parametrize("variant", ["FP16_APPROX", "BF16_APPROX", "FP16S_APPROX", "BF16S_APPROX"])
@pytest.mark.parametrize("payoff,scheme,level,method", [(W.EURO, W.EULER, 2, 1), (W.ASIAN, W.MILSTEIN, 3, 1),
                                                        (W.LOOKBACK, W.EULER, 5, 3), (W.DIGITAL, W.MILSTEIN, 8, 1)])
def test_two_samples_per_thread(m, variant, payoff, scheme, level, method):
    """Above 128 x 608 samples a thread has two or more; the parts give it one."""
    P = m.make_params(W.params(payoff=payoff, scheme=scheme), method=method)
    for N in (128 * 608 + 1, 128 * 608 * 2 + 131, 128 * 608 * 3 - 77):
        s = m.mlmc_level(level, N, P, getattr(m, variant), 7, 11)
        _same(s, _parts(m, level, N, P, getattr(m, variant), 7, 11, 70_001), N)


@pytest.mark.parametrize("level,variant,pack", [(1, "FIXED_APPROX", 1), (0, "FIXED_APPROX", 1), (1, "FP16_APPROX", 0),
                                                (0, "FP32_EXACT", 0), (2, "NESTED_CORR_FIXED", 0)])
def test_larger_chunks(m, level, variant, pack):
    """More than 24 chunks of the default size per SM take larger ones; the parts do not."""
    P = m.make_params(W.params(), rng_pack=pack)
    per = 128 * (256 >> level) // (3 if pack else 1) * (3 if pack else 1)   # samples per default chunk, nearly
    for N in (24 * 152 * per + per, 60 * 152 * per + 12_345):
        s = m.mlmc_level(level, N, P, getattr(m, variant), 9, 1)
        _same(s, _parts(m, level, N, P, getattr(m, variant), 9, 1, 12 * 152 * per), N)


@pytest.mark.parametrize("pack", [0, 1])
@pytest.mark.parametrize("frac", [14, 21])
def test_level0_values(m, frac, pack):
    """Narrow S: a thread's sums in 64 bits to the end; wide S: added up by group."""
    p = W.params(payoff=W.EURO)
    f = W.default_format(p, 0)
    f["f"][6] = frac
    P = m.make_params(p, formats=[f], rng_pack=pack)
    N = 400_003
    s = m.mlmc_level(0, N, P, m.FIXED_APPROX, 3, 2)
    t, _ = m.mlmc_level_dump(0, N, P, m.FIXED_APPROX, 3, 2)
    _same(s, t, N)


@pytest.mark.parametrize("payoff", [W.EURO, W.DIGITAL, W.ASIAN, W.LOOKBACK])
@pytest.mark.parametrize("scheme", [W.EULER, W.MILSTEIN])
@pytest.mark.parametrize("level", [1, 2, 4])
def test_lazy_corrections_that_saturate(m, payoff, scheme, level):
    """S limited to 128 (S0 = 100): corrections whose S leaves it run again with the clamps,
    as the record-writing kernel runs them all."""
    p = W.params(payoff=payoff, scheme=scheme)
    fmts = [W.default_format(p, lev) for lev in range(level + 1)]
    for f in fmts:
        f["e"][6] = 7
    P = m.make_params(p, formats=fmts)
    N = 20_011
    s = m.mlmc_level(level, N, P, m.NESTED_CORR_FIXED, 21, 4)
    t, rec = m.mlmc_level_dump(level, N, P, m.NESTED_CORR_FIXED, 21, 4)
    assert s["saturations"] == t["saturations"] == int(rec["sat"].sum()) and s["saturations"] > 100
    _same(s, t, N)


@pytest.mark.parametrize("level,N", [(0, 1), (0, 129), (1, 127), (2, 128), (3, 257), (6, 608 * 128 + 1), (7, 5000), (10, 200)])
def test_sensitivity_batches(m, level, N):
    """Statistics of [0, N) from those of two ranges of it."""
    P = m.make_params(W.params())
    a = m.mlmc_sensitivities(level, N, P, 5, 0, per_instance=True)
    n1 = max(1, N // 3)
    parts = [(n, m.mlmc_sensitivities(level, n, P, 5, at, per_instance=True)) for at, n in ((0, n1), (n1, N - n1)) if n]
    for k in ("A", "inst"):
        want = sum(n * np.asarray(s[k]) for n, s in parts) / N
        assert np.all(np.abs(np.asarray(a[k]) - want) <= 1e-11 * np.abs(want) + 1e-300), k
    assert np.array_equal(a["maxabs"], np.max([s["maxabs"] for _, s in parts], axis=0))
