"""Plain FP64 sums of many rows: constant columns, whose roundings do not average out, on one block, so that a
thread's rows are as many as a whole grid's of 600 times as many rows.

The bound is the number of additions one after another on the way to a sum, half an ulp each: at most 256 in a
thread's first sum and its first rows (256) before that is emptied, its rows over 128 in its second, the
tree over at most 128 slices of rows and a slot's last steps.  A thread's rows: p columns make `tiles` tiles of 2 x 2,
and a block of 128 threads at least (256 from eight tiles on) deals its rows to as many threads a tile."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")

N = 3_000_001


@pytest.mark.parametrize("p", [1, 2, 5, 8, 9, 11, 12])
@pytest.mark.parametrize("mode", [G.STATS_FP64, G.STATS_FP64_SHIFTED])
def test_blocked_sums(p, mode):
    value = [0.1 * (j + 1) + 0.7 for j in range(p)]
    cols = [torch.full((N,), v, dtype=torch.float64, device="cuda") for v in value]
    if mode == G.STATS_FP64_SHIFTED:  # the pivot: zero, from the first 64 rows
        for c in cols:
            c[:64] = 0.0
    n = N - (64 if mode == G.STATS_FP64_SHIFTED else 0)
    ctx = G.stats_init(G.Config([G.STATS_F64] * p, mode))
    G.stats_set_grid(ctx, 1)
    G.stats_accumulate(ctx, cols, N)
    raw = G.stats_raw(ctx)
    tiles = (p + 1) // 2 * ((p + 1) // 2 + 1) // 2
    rows = N / (128 // tiles) if tiles < 8 else N / (256 // tiles)
    bound = (256 + 256 + rows / 128 + 16) * 2.0 ** -53
    for j in range(p):
        assert abs(Fraction(float(raw.s[j])) / (n * Fraction(value[j])) - 1) <= bound
        for k in range(j, p):
            assert abs(Fraction(float(raw.S[j, k])) / (n * Fraction(value[j]) * Fraction(value[k])) - 1) <= bound
