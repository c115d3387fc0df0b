"""A batch's decompositions are shared by 4, 2 or 1 blocks, by their number: the same bits however many
there are, at the counts where the share changes on a 152-SM device, with an undefined one among them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")

WIDTHS = [24, 25, 31, 32, 33, 47, 48, 49, 63, 64]


def context(p, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((p, 3 * p)) * np.linspace(1.0, 3.0, p)[:, None] + 0.3 * rng.standard_normal(3 * p)
    cols = [torch.from_numpy(np.ascontiguousarray(c)).cuda() for c in x]
    ctx = G.stats_init(G.Config([G.STATS_F64] * p, G.STATS_FP64_SHIFTED))
    G.stats_accumulate(ctx, cols, x.shape[1])
    return ctx


@pytest.fixture(scope="module")
def singles():
    ctxs = [context(p, p) for p in WIDTHS]
    return ctxs, [G.stats_finalize_batched([c])[0] for c in ctxs]


@pytest.mark.parametrize("count", [2, 76, 77, 152, 153])
def test_same_bits_for_any_count(singles, count):
    ctxs, ref = singles
    out = G.stats_finalize_batched([ctxs[i % len(ctxs)] for i in range(count)])
    for i, an in enumerate(out):
        r = ref[i % len(ctxs)]
        assert np.array_equal(an.evals, r.evals) and np.array_equal(an.evecs, r.evecs)
    for an, p in zip(ref, WIDTHS):
        assert np.abs(an.evecs @ an.evecs.T - np.eye(p)).max() <= 1e-12
        scale = np.abs(an.cov).max() * p ** 0.5
        assert np.abs(an.evecs @ an.cov @ an.evecs.T - np.diag(an.evals)).max() <= 1e-12 * scale


def test_undefined_among_others(singles):
    ctxs, ref = singles
    flat = G.stats_init(G.Config([G.STATS_F64] * 30, G.STATS_FP64_SHIFTED))
    G.stats_accumulate(flat, [torch.full((50,), 2.0, dtype=torch.float64, device="cuda")] * 30, 50)
    out = G.stats_finalize_batched([ctxs[9], flat, ctxs[0]], 1)
    assert np.all(np.isnan(out[1].evals))
    assert np.all(np.isfinite(out[0].evals)) and np.all(np.isfinite(out[2].evals))
