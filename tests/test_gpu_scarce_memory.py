"""The error model's device workspace where the device has little room: fewer CTAs
instead of a refusal, the kept part given back to the library's other
allocations, and no error left behind for the call after a refusal."""
import numpy as np
import pytest

from paper_2502_07123_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def m():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2502_07123_gb300 import mlmc
    return mlmc


@pytest.fixture
def leave():
    """leave(n): allocates all but about n bytes of the device's free memory until the test ends."""
    import torch
    held = []

    def fill(n):
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        if free > n:
            held.append(torch.empty(free - n, dtype=torch.uint8, device="cuda"))

    yield fill
    held.clear()
    torch.cuda.empty_cache()


@pytest.mark.parametrize("level,N,room", [(10, 50_000, 320 * MB), (7, 90_001, 160 * MB)])
def test_statistics_with_fewer_ctas(m, leave, level, N, room):
    """The whole grid's tapes take 1.07 GB at level 10 and 239 MB at level 7."""
    P = m.make_params(W.params())
    want = m.mlmc_sensitivities(level, N, P, 5, per_instance=True)
    leave(room)
    got = m.mlmc_sensitivities(level, N, P, 5, per_instance=True)
    # two orders of the same FP64 sums: a few hundred terms of one sign each
    for k in ("A", "B", "inst"):
        np.testing.assert_allclose(got[k], want[k], rtol=1e-12, err_msg=k)
    np.testing.assert_array_equal(got["maxabs"], want["maxabs"])
    assert got["mean"] == pytest.approx(want["mean"], rel=1e-9, abs=1e-12)


def test_no_error_left_by_a_refusal(m, leave):
    P = m.make_params(W.params())
    m.mlmc_level(3, 1000, P, m.FP32_EXACT, 1)
    leave(64 * MB)
    with pytest.raises(m.MLMCError) as e:   # several GB of slots
        m.Engine(max_slots=200_000, max_level=10)
    assert e.value.status == m.ENOMEM
    m.mlmc_level(3, 1000, P, m.FP32_EXACT, 1)


def test_kept_workspace_is_given_back(m, leave):
    """117 MB are kept after a level-6 call; an engine that needs them gets them."""
    P = m.make_params(W.params())
    m.mlmc_sensitivities(6, 100_001, P, 5)
    leave(64 * MB)
    eng = m.Engine(max_slots=3000, max_level=10)
    assert eng.stats()["slots"] == 3000
    eng.close()
