"""How the fragment pass deals a launch's stages to the SMs: row counts where a table fills one stage, one
stage an SM, one shortest chunk an SM, and one more or less.
Against FP64 on the same values, to the modes' stated covariance error (2e-6 of the deviations); the
column means to that of one FP32 pivot and exact differences (1e-9 of the deviations)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")

ROWS = {8: 2048, 16: 1024, 24: 240, 40: 240}  # rows of a stage


def columns(p, n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn((p, n), generator=g, device="cuda")
    x += 0.5 * x[0] + 100.0
    return [c.clone() for c in x]  # apart: no tensor copies of a block


def check(an, cols):
    x = torch.stack(cols).double()
    mean = x.mean(dim=1)
    x -= mean[:, None]
    cov = (x @ x.t() / (x.shape[1] - 1)).cpu().numpy()
    sd = np.sqrt(np.diag(cov))
    assert np.abs((an.cov - cov) / np.outer(sd, sd)).max() <= 2e-6
    assert np.abs((an.mean - mean.cpu().numpy()) / sd).max() <= 1e-9


@pytest.mark.parametrize("mode", [G.STATS_BF16X3, G.STATS_BF16X4])
@pytest.mark.parametrize("p", sorted(ROWS))
@pytest.mark.parametrize("stages", [1, 2, 151, 152, 153, 31 * 152, 32 * 152, 33 * 152])
def test_rows_around_the_split(mode, p, stages):
    for n in (stages * ROWS[p] - 1, stages * ROWS[p] + 1):
        cols = columns(p, n, stages)
        with G.stats_init(G.Config([G.STATS_F32] * p, mode)) as ctx:
            G.stats_accumulate(ctx, cols, n)
            check(G.stats_finalize(ctx), cols)
