"""STATS_FP32 near the end of FP32's range: sums of squares that FP32 holds for the rows dealt to a thread, but
not for a block's or for all of them.  64 x 64 tiles on four blocks an SM, 4096 rows a block at least, set
what has to be held: sums up to FP32's range times that number of blocks are finite and accurate.

Entries of +-sigma with a pivot of zero: every variance is known but for the sample's mean.  A sum in
FP32 pairs keeps 1e-7 of its size or better; 1e-6 of sigma^2 is asked."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")

N = 430_001


def dealt(p):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = (p + 63) // 64 * ((p + 63) // 64 + 1) // 2
    return min(N // 4096, (4 * sms + tiles - 1) // tiles)


@pytest.mark.parametrize("p", [1, 2, 12, 33, 64, 100, 128, 176, 180, 192, 224, 252, 256])
def test_sums_past_a_blocks_range(p):
    sigma = np.float32((0.9 * 3.4e38 * dealt(p) / N) ** 0.5)
    g = torch.Generator(device="cuda")
    g.manual_seed(p)
    s = torch.randint(0, 2, (p, N), generator=g, device="cuda", dtype=torch.int8) * 2 - 1
    s[:, 0:64:2], s[:, 1:64:2] = 1, -1
    cols = [(row.float() * float(sigma)) for row in s]
    ctx = G.stats_init(G.Config([G.STATS_F32] * p, G.STATS_FP32))
    G.stats_accumulate(ctx, cols, N)
    raw, an = G.stats_raw(ctx), G.stats_finalize(ctx)
    S = s.double() @ s.double().t()
    total = s.sum(dim=1, dtype=torch.float64)
    want = (S - torch.outer(total, total) / N).cpu().numpy() / (N - 1)
    unit = float(sigma) ** 2
    assert np.abs(raw.S / unit - S.cpu().numpy()).max() <= 1e-6 * N
    assert np.abs(an.cov / unit - want).max() <= 1e-6
    assert np.abs(an.corr - want / np.sqrt(np.outer(np.diag(want), np.diag(want)))).max() <= 1e-6
