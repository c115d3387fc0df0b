"""The CUDA-core passes (FP32-core; FP64 raw and shifted) at the edges of their cuts: widths around
the micro-tiles, row counts around stages, columns off 16-byte alignment, and every column type.

Reference: the same sums in numpy.  Bounds: a sum of m products accumulated in any order with
unit roundoff u is off by at most (m + 2) u times the sum of the products' magnitudes (m rows of a
chain; for FP32 chains of at most 64 rows, then pairs, plus the two roundings of x - c).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")

NP = {G.STATS_I16: np.int16, G.STATS_I32: np.int32, G.STATS_I64: np.int64, G.STATS_F32: np.float32,
      G.STATS_F64: np.float64}


def columns(dtypes, n, seed):
    rng = np.random.default_rng(seed)
    z = rng.standard_normal((len(dtypes), n))
    z[1:] += 0.5 * z[:1]
    return [(3.0 + z[j]).astype(NP[d]) if d in (G.STATS_F32, G.STATS_F64) else
            np.rint(50 + 200 * z[j]).astype(NP[d]) for j, d in enumerate(dtypes)]


def on_device(cols, offset):
    """Device copies; offset: elements by which a column starts after its 256-byte aligned buffer."""
    out = []
    for c in cols:
        buf = torch.empty(c.size + 8, dtype=torch.from_numpy(c[:1]).dtype, device="cuda")
        out.append(buf[offset:offset + c.size].copy_(torch.from_numpy(c)))
    return out


def check(dtypes, n, mode, seed, offset=0, parts=1, grid=0):
    cols = columns(dtypes, n, seed)
    dev = on_device(cols, offset)
    with G.stats_init(G.Config(dtypes, mode)) as ctx:
        if grid:
            G.stats_set_grid(ctx, grid)
        cut = [n * i // parts for i in range(parts + 1)]
        for a, b in zip(cut, cut[1:]):
            G.stats_accumulate(ctx, [d[a:b] for d in dev], b - a)
        raw = G.stats_raw(ctx)
        first = cut[1]
    assert raw.n == n
    X = np.stack([c.astype(np.float64) for c in cols])
    c = X[:, :min(64, first)].mean(axis=1)
    R = X - c[:, None] if mode != G.STATS_FP64 else X
    mag = np.abs(R) @ np.abs(R).T
    # FP64 rounding of the whole, of the reference and of the pivot terms that raw sums add back
    full = np.abs(X) @ np.abs(X).T + n * np.outer(np.abs(c), np.abs(c))
    u = (68 * 2.0 ** -24) if mode == G.STATS_FP32 else n * 2.0 ** -53
    sums = np.abs(R).sum(axis=1) * u + (np.abs(X).sum(axis=1) + n * np.abs(c)) * n * 2.0 ** -52
    assert np.all(np.abs(raw.s - X.sum(axis=1)) <= sums)
    # S = S' + c s'^T + s' c^T + n c c^T: the sums' errors come back times the pivot
    bound = mag * u + full * n * 2.0 ** -52
    if mode != G.STATS_FP64:
        bound += np.outer(np.abs(c), sums) + np.outer(sums, np.abs(c))
    assert np.all(np.abs(raw.S - X @ X.T) <= bound)


@pytest.mark.parametrize("n", [1, 65, 2047, 40_003])
@pytest.mark.parametrize("p", [1, 2, 8, 9, 33, 64, 100, 129, 255, 256])
def test_fp32_core_widths_and_rows(p, n):
    check([G.STATS_F32] * p, n, G.STATS_FP32, 10 * p + n)


@pytest.mark.parametrize("p,offset,parts,grid", [(5, 1, 1, 0), (40, 3, 3, 0), (72, 0, 4, 7), (130, 2, 1, 1)])
def test_fp32_core_alignment_calls_and_grids(p, offset, parts, grid):
    check([G.STATS_F32] * p, 10_007, G.STATS_FP32, p, offset, parts, grid)


@pytest.mark.parametrize("offset", [0, 1])
def test_fp32_core_column_types(offset):
    check([G.STATS_I16, G.STATS_F32, G.STATS_I32, G.STATS_F64, G.STATS_I64] * 3, 5_001, G.STATS_FP32, 3, offset)


@pytest.mark.parametrize("n", [1, 33, 4_099, 40_003])
@pytest.mark.parametrize("p", [1, 2, 3, 8, 12, 13, 16, 31, 48, 65, 127, 128, 200, 256])
@pytest.mark.parametrize("mode", [G.STATS_FP64, G.STATS_FP64_SHIFTED])
def test_fp64_core_widths_and_rows(mode, p, n):
    check([G.STATS_F64] * p, n, mode, 7 * p + n)


@pytest.mark.parametrize("p,parts,grid", [(14, 3, 0), (50, 1, 5), (140, 2, 1)])
def test_fp64_core_calls_and_grids(p, parts, grid):
    check([G.STATS_F64] * p, 10_007, G.STATS_FP64_SHIFTED, p, 1, parts, grid)


@pytest.mark.parametrize("mode", [G.STATS_FP64, G.STATS_FP64_SHIFTED])
def test_fp64_core_column_types(mode):
    for k in (1, 2, 3):
        check([G.STATS_I16, G.STATS_F32, G.STATS_I32, G.STATS_F64, G.STATS_I64] * k, 5_001, mode, 4, 1)
