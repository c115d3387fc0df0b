"""Reals of a generic exact plan: fixed point to nearest, ties to even (as Table 1's), subnormal values
among them; sums bit for bit against rational arithmetic."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")


def fixed(x, e, signed):
    """x rounded to a multiple of 2^(e - P), ties to even."""
    unit = Fraction(2) ** (e - (54 if signed else 55))
    q = Fraction(float(x)) / unit
    n, r = divmod(q.numerator, q.denominator)
    twice = 2 * r - q.denominator
    if twice > 0 or (twice == 0 and n % 2):
        n += 1
    return n * unit


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("lo,hi", [(-1.0, 1.0), (0.0, 1.0), (-4096.0, 4096.0), (0.0, 1e-300),
                                   (-1e-305, 1e-305)])
def test_ties_and_subnormals(lo, hi, offset):
    e, signed = int(np.frexp(max(abs(lo), hi))[1]), lo < 0
    unit = Fraction(2) ** (e - (54 if signed else 55))
    rng = np.random.default_rng(3)
    x = [0.0, hi, 5e-324 if hi >= 5e-324 else 0.0]
    for k in range(1, 400):  # halves of the unit and values beside them, where a double has them
        v = float(Fraction(2 * k + 1, 2) * unit)
        x += [v, np.nextafter(v, 0.0), np.nextafter(v, hi)]
    x += list(lo + (hi - lo) * rng.random(300))
    x = np.array([min(max(v, 0.0), hi) for v in x])
    if signed:
        x = np.concatenate([x, -x])
    n = len(x)
    buf = torch.zeros(n + 8, dtype=torch.float64, device="cuda")
    ones = torch.ones(n + 8, dtype=torch.int16, device="cuda")
    buf[offset:offset + n] = torch.from_numpy(x)
    with G.stats_init(G.Config([G.STATS_I16, G.STATS_F64], G.STATS_EXACT, None, [0.0, lo], [3.0, hi])) as ctx:
        for i in range(n):  # one row a call shows each value's rounding
            if i >= 60 and i % 37:
                continue
            G.stats_reset(ctx)
            G.stats_accumulate(ctx, [ones[offset:], buf[offset + i:]], 1)
            assert Fraction(float(G.stats_raw(ctx).s[1])) == fixed(x[i], e, signed), (i, x[i])
        G.stats_reset(ctx)
        G.stats_accumulate(ctx, [ones[offset:], buf[offset:]], n)
        total = sum((fixed(v, e, signed) for v in x), Fraction(0))
        assert float(G.stats_raw(ctx).s[1]) == float(total)
