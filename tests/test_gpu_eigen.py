"""The eigen-solvers at the orders where they change (one block up to 23 and, in a batch, 64 columns; the
grid; FP32 rotations in one block up to 96, over the grid above) and on the spectra that leave the
refinement for FP64 rotations: equal and nearly equal eigenvalues, zero variances, columns of very
different units, values whose squares leave FP64's range.

Checked on the returned matrix itself: orthonormal vectors, a diagonal V M V^T, and the eigenvalues
LAPACK gives, all to O(p eps) of the matrix's norm; for graded matrices, whose small eigenvalues are
far below that, each eigenvalue against the oracle's Jacobi."""
import numpy as np
import pytest

import oracle as O
from paper_2604_23826_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")


def contexts(X, count=1):
    cols = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in X]
    ctxs = [G.stats_init(G.Config([G.STATS_F64] * len(X), G.STATS_FP64_SHIFTED)) for _ in range(count)]
    for c in ctxs:
        G.stats_accumulate(c, cols, X.shape[1])
    return ctxs


def check(an, M):
    p, scale = len(M), np.abs(M).max() * len(M) ** 0.5
    assert np.abs(an.evecs @ an.evecs.T - np.eye(p)).max() <= 1e-12
    assert np.abs(an.evecs @ M @ an.evecs.T - np.diag(an.evals)).max() <= 1e-12 * max(scale, 1e-300)
    assert np.all(np.diff(an.evals) <= 0)
    assert np.abs(an.evals - np.linalg.eigvalsh(M)[::-1]).max() <= 4e-15 * p * scale
    big = an.evecs[np.arange(p), np.argmax(np.abs(an.evecs), axis=1)]
    assert np.all(big > 0)


def both(X, pca_on=0):
    """The single and the batched result of the same table."""
    a, b = contexts(X, 2)
    single = G.stats_finalize(a, pca_on)
    batch = G.stats_finalize_batched([a, b], pca_on)
    assert np.array_equal(batch[0].evecs, batch[1].evecs)
    assert np.array_equal(single.cov, batch[0].cov) and np.array_equal(single.corr, batch[0].corr, equal_nan=True)
    if len(X) < 24:
        assert np.array_equal(single.evals, batch[0].evals) and np.array_equal(single.evecs, batch[0].evecs)
    return single, batch[0]


@pytest.mark.parametrize("p", [1, 2, 3, 11, 22, 23, 24, 25, 44, 45, 63, 64, 65, 80, 96, 97, 128, 160, 193, 256])
@pytest.mark.parametrize("pca_on", [0, 1])
def test_orders(p, pca_on):
    L, mu = inputs.wide_factor(100 + p, p)
    X = inputs.gen_correlated_host(40 * p + 500, L, mu, seed=p)
    for an in both(X, pca_on):
        check(an, an.corr if pca_on else an.cov)


@pytest.mark.parametrize("p", [6, 23, 33, 64, 100, 130])
def test_close_and_equal_eigenvalues(p):
    """Orthogonal columns of equal, nearly equal and zero variance, mixed by one rotation of pairs."""
    rng = np.random.default_rng(p)
    q, _ = np.linalg.qr(rng.standard_normal((400 + p, p)))
    q -= q.mean(axis=0)
    sd = np.repeat(np.linspace(1.0, 2.0, (p + 2) // 3), 3)[:p]
    sd[1::6] *= 1 + 1e-9
    sd[-2:] = 0.0
    X = (q * sd).T * 20.0 + 3.0
    X[0] += 0.5 * X[p // 2]
    for an in both(X):
        check(an, an.cov)


@pytest.mark.parametrize("p", [5, 12, 23])
def test_graded_columns(p):
    """Correlated columns whose units span four decades, the eigenvalues eight or more: every eigenvalue to 1e-9 of itself."""
    L, mu = inputs.wide_factor(7, p)
    X = inputs.gen_correlated_host(3_000, L, np.zeros(p), seed=3) * 10.0 ** np.linspace(2, -2, p)[:, None]
    for an in both(X):
        ev, _ = O.jacobi(an.cov)
        assert np.abs(an.evals / ev - 1.0).max() <= 1e-9
        assert np.abs(an.evecs @ an.evecs.T - np.eye(p)).max() <= 1e-12


@pytest.mark.parametrize("scale", [1e-71, 1e-60, 1e60, 1e72])
@pytest.mark.parametrize("p", [4, 30, 100])
def test_extreme_scales(p, scale):
    L, mu = inputs.wide_factor(9, p)
    X = inputs.gen_correlated_host(2_000, L, np.zeros(p), seed=4)
    (ctx,) = contexts(X * scale)
    an = G.stats_finalize(ctx)
    ref = G.stats_finalize(contexts(X)[0])
    unit = an.evals.max()
    assert unit > 0 and np.isfinite(unit)
    # a matrix of the same shape: the eigenvalues over the largest, to the data's own rounding
    keep = np.abs(ref.evals) > 1e-9 * ref.evals.max()
    assert np.abs(an.evals[keep] / unit - ref.evals[keep] / ref.evals.max()).max() <= 1e-12
    assert np.abs(an.evecs @ an.evecs.T - np.eye(p)).max() <= 1e-12


@pytest.mark.parametrize("p", [3, 40])
def test_zero_matrix(p):
    for an in both(np.full((p, 100), 2.5)):
        assert np.all(an.evals == 0) and np.array_equal(np.abs(an.evecs), np.eye(p))


@pytest.mark.parametrize("p", [24, 40, 64, 65, 100, 256])
def test_rank_deficient(p):
    """Fewer rows than columns, and every column twice: half of the eigenvalues are zero."""
    rng = np.random.default_rng(p)
    for X in (rng.standard_normal((p, p // 2)), np.repeat(rng.standard_normal((p - p // 2, 4 * p)), 2, axis=0)[:p]):
        for an in both(X):
            check(an, an.cov)
