"""Eigenpairs of columns of very different units, in any order: cold, in a batch, and seeded by the vectors of
the first half of the rows; with well separated eigenvalues, and with close ones among the small ones.

The small eigenvalues lie far below the rounding of the largest, so nothing here compares to the matrix's
norm: V M V^T has to be diagonal in each pair's own units, which bounds every eigenvalue's relative
error and, over the relative gap, every vector's.  The bound: a product X^T M X rounds by at most
2 p eps sum |x_ki| |m_kl| |x_lj|, |m_kl| <= sqrt(m_kk m_ll), and sum_k sqrt(m_kk) |x_ki| is at most
sqrt(p lambda_i / lambda_min(corr)); once for the solver's own products, once for this check's."""
import numpy as np
import pytest

from paper_2604_23826_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")

N = 3_000


def units(p, decades, rng):
    return rng.permutation(10.0 ** np.linspace(decades / 2, -decades / 2, p))


def separated(p, decades):
    rng = np.random.default_rng([p, decades])
    L, _ = inputs.wide_factor(7, p)
    return inputs.gen_correlated_host(N, L, np.zeros(p), seed=3) * units(p, decades, rng)[:, None]


def close(p, width):
    """Groups of three columns with eigenvalues equal but for `width`, the groups' units over six decades."""
    rng = np.random.default_rng([p, int(1 / width)])
    x = rng.standard_normal((N, p))
    x = np.linalg.qr(x - x.mean(axis=0))[0].T * (1 + width * rng.random(p))[:, None]
    scale = np.repeat(10.0 ** np.linspace(3, -3, (p + 2) // 3), 3)[:p]
    for g in range(0, p - 2, 3):
        x[g:g + 3] = np.linalg.qr(rng.standard_normal((3, 3)))[0] @ x[g:g + 3]
    return (x * scale[:, None])[rng.permutation(p)]


def context(X, n):
    ctx = G.stats_init(G.Config([G.STATS_F64] * len(X), G.STATS_FP64_SHIFTED))
    G.stats_accumulate(ctx, [torch.from_numpy(np.ascontiguousarray(x[:n])).cuda() for x in X], n)
    return ctx


def check(an):
    p, M = len(an.cov), an.cov
    sd = np.sqrt(np.diag(M))
    bound = 4 * p * p * 2.0 ** -53 / np.linalg.eigvalsh(M / np.outer(sd, sd))[0]
    assert np.all(an.evals > 0) and np.all(np.diff(an.evals) <= 0)
    assert np.abs(an.evecs @ an.evecs.T - np.eye(p)).max() <= 1e-12
    R = (an.evecs @ M @ an.evecs.T - np.diag(an.evals)) / np.sqrt(np.outer(an.evals, an.evals))
    assert np.abs(R).max() <= bound


def all_ways(X):
    a, b, half = context(X, N), context(X, N), context(X, N // 2)
    seed = G.stats_finalize(half).evecs
    yield G.stats_finalize(a)
    yield from G.stats_finalize_batched([a, b])
    yield G.stats_finalize_warm(a, 0, seed)


@pytest.mark.parametrize("p", [3, 12, 23, 24, 25, 40, 64, 65, 100, 256])
@pytest.mark.parametrize("decades", [4, 6, 8])
def test_units(p, decades):
    for an in all_ways(separated(p, decades)):
        check(an)


@pytest.mark.parametrize("p", [12, 24, 40, 65, 100])
@pytest.mark.parametrize("width", [1e-4, 1e-7])
def test_close_eigenvalues_of_small_units(p, width):
    for an in all_ways(close(p, width)):
        check(an)


@pytest.mark.parametrize("p", [24, 25, 31, 32, 33, 40, 47, 48, 49, 56, 63, 64])
def test_batched_results_come_from_the_refinement(p):
    """Well separated eigenvalues: the refinement of a batch adds the same products in the same order as the
    grid's, after FP32 rotations of the same order, so its results are a single call's bits; FP64 rotations
    (what a batch falls back to) leave others."""
    X = separated(p, 0)
    a, b = context(X, N), context(X, N)
    single = G.stats_finalize(a)
    check(single)
    for an in G.stats_finalize_batched([a, b]):
        assert np.array_equal(an.evals, single.evals) and np.array_equal(an.evecs, single.evecs)


def test_snapshots_agree_with_cold_results():
    """A stream's seeded snapshots against the cold result of the same rows, vector by vector."""
    X = separated(12, 6)
    with G.StreamingAnalysis(G.Config([G.STATS_F64] * 12, G.STATS_FP64_SHIFTED)) as s:
        for r in range(0, N, 1000):
            s.update([torch.from_numpy(np.ascontiguousarray(x[r:r + 1000])).cuda() for x in X], 1000)
            an, cold = s.snapshot(), G.stats_finalize(s.ctx)
            assert np.array_equal(an.cov, cold.cov)
            assert np.abs(an.evals / cold.evals - 1.0).max() <= 1e-9
            assert np.abs(an.evecs - cold.evecs).max() <= 1e-9


@pytest.mark.parametrize("p,most", [(64, 20), (256, 26)])
def test_clusters_go_on_from_the_refined_basis(p, most):
    """Four clusters of width 1e-6: FP32 and FP64 sweeps together, fewer than FP32's and those that FP64
    rotations from the identity take (24 and 32); the results to rounding."""
    rng = np.random.default_rng(p)
    x = rng.standard_normal((3 * p, p))
    k = np.arange(p)
    x = np.linalg.qr(x - x.mean(axis=0))[0] * np.sqrt((1.0 + k % 4) * (1 + 1e-6 * (k // 4) / (p / 4)))
    X = (x @ np.linalg.qr(rng.standard_normal((p, p)))[0].T).T
    an = G.stats_finalize_warm(context(X, 3 * p))
    scale = np.abs(an.evals).max()
    assert 0 < an.sweeps <= most
    assert np.abs(an.evecs @ an.evecs.T - np.eye(p)).max() <= 1e-12
    assert np.abs(an.evecs @ an.cov @ an.evecs.T - np.diag(an.evals)).max() <= 1e-13 * scale


@pytest.mark.parametrize("p", [6, 12, 23, 24, 40, 64, 100, 256])
def test_units_and_repeated_columns(p):
    """Half of the eigenvalues zero, at every unit: their rounding, eps of the repeated columns' variance, hides the
    eigenvalues of smaller units, so some pairs go through FP64 rotations.  The same bound, by the vectors' own
    sums: it holds for what ends in the refinement, so for all but batches above 64 columns (FP64 rotations
    alone, whose intermediate vectors it says nothing about)."""
    rng = np.random.default_rng(p)
    L, _ = inputs.wide_factor(p, p)
    X = inputs.gen_correlated_host(N, L, np.zeros(p), seed=1) * 10.0 ** rng.uniform(-4, 4, p)[:, None]
    X[p // 2:p // 2 * 2] = X[:p // 2]
    X = X[rng.permutation(p)]
    warm = G.stats_finalize_warm(context(X, N))
    assert 0 < warm.sweeps < 45
    single, *batch, seeded = all_ways(X)
    for an in (warm, single, seeded, *(batch if p <= 64 else ())):
        s = np.abs(an.evecs) @ np.sqrt(np.diag(an.cov))
        assert np.abs(an.evecs @ an.evecs.T - np.eye(p)).max() <= 1e-12
        R = an.evecs @ an.cov @ an.evecs.T - np.diag(an.evals)
        assert np.all(np.abs(R) <= 4 * p * 2.0 ** -53 * np.outer(s, s))
