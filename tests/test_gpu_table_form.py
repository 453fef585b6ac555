"""Shared-memory tables of 4 and 8 bytes an index: the same item with and without
per-sample records (8 and 4 bytes, through the cache of built items), tables of
several sizes one after another in the same kernel, and work lists that mix both
forms in one launch."""
import pytest

from paper_2502_07123_gb300 import workloads as W
from tests.test_gpu_chunk_forms import _same

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


@pytest.mark.parametrize("variant", ["FIXED_APPROX", "NESTED_CORR_FIXED"])
@pytest.mark.parametrize("payoff,scheme", [(W.EURO, W.EULER), (W.ASIAN, W.EULER), (W.LOOKBACK, W.MILSTEIN)])
@pytest.mark.parametrize("level", [0, 1, 4])
def test_records_and_sizes_in_turn(m, variant, payoff, scheme, level):
    p, v, N = W.params(payoff=payoff, scheme=scheme), getattr(m, variant), 5003
    P = {d: m.make_params(p, d=d, method=meth) for d, meth in ((12, 1), (3, 1), (10, 3), (14, 1), (11, 1))}
    for d in (12, 3, 10, 14, 11, 12):
        first = m.mlmc_level(level, N, P[d], v, 8, 5)
        rec, _ = m.mlmc_level_dump(level, N, P[d], v, 8, 5, stream=1 if variant == "FIXED_APPROX" else 0)
        again = m.mlmc_level(level, N, P[d], v, 8, 5)
        _same(first, rec, N)
        _same(again, rec, N)


@pytest.mark.parametrize("d", [10, 12])
@pytest.mark.parametrize("sigma", [0.2, 0.6])
def test_forms_in_one_launch(m, d, sigma):
    """sigma 0.2: 4 bytes throughout; 0.6: most levels keep the 8-byte pairs (family 17)."""
    items = []
    for payoff in (W.EURO, W.DIGITAL):
        for s in (sigma, 0.2):
            P = m.make_params(W.params(payoff=payoff, sigma=s), d=d, request=int(10 * s) + payoff)
            items += [dict(params=P, level=lev, variant=v, N=20_003 >> lev)
                      for lev in range(7) for v in (m.FIXED_APPROX, m.NESTED_CORR_FIXED)]
    plan = m.Plan(items, 6)
    families = {plan.launch_info(k)[0] for k in range(plan.info()["kernels"])}
    assert (24 if sigma == 0.2 else 17) in families
    for it, r in zip(items, m.mlmc_run(items, 6)):
        _same(r, m.mlmc_level(it["level"], it["N"], it["params"], it["variant"], 6), it["N"])
