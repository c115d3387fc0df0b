"""gram32_min_chunk: a caller's shortest chunk holds also where it leaves CTAs without one (the rows are then
added in fewer partial sums, whose last bits differ); the default gives way there."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")
from paper_2604_23826_gb300 import tune  # noqa: E402


@pytest.mark.parametrize("p", [8, 13, 32])
def test_a_callers_chunk_holds(p):
    n = 300_000
    g = torch.Generator(device="cuda")
    g.manual_seed(p)
    cols = list(torch.rand((p, n), generator=g, device="cuda"))

    def S(min_chunk):
        G.stats_set_batch_tuning(p, G.STATS_BF16X3, dict(tune.DEFAULT, gram32_min_chunk=min_chunk))
        ctx = G.stats_init(G.Config([G.STATS_F32] * p, G.STATS_BF16X3))
        G.stats_accumulate_batched([ctx], [cols], [n])
        return G.stats_raw(ctx).S

    try:
        dealt, one, also_one, default = S(1), S(65536), S(60000), S(tune.DEFAULT["gram32_min_chunk"])
    finally:
        G.stats_set_batch_tuning(p, G.STATS_BF16X3, tune.DEFAULT)
    assert np.array_equal(one, also_one)  # one chunk holds all rows either way
    assert not np.array_equal(one, dealt)
    assert not np.array_equal(one, default)
    assert np.abs(one / dealt - 1).max() <= 1e-6 and np.abs(default / dealt - 1).max() <= 1e-6
