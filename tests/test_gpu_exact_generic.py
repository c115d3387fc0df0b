"""The exact pass's generic converter over the forms a digit plan takes: every column type, field
width and sign at shifting byte offsets, reals at the edges of their fixed point, values at and past
the ends of their fields.  Integers bit for bit; reals against exact rational sums: each value is
rounded to a fixed point of 2^-55 of its range (2^-54 when signed), half a unit at most."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")

NP = {G.STATS_I16: np.int16, G.STATS_I32: np.int32, G.STATS_I64: np.int64, G.STATS_F32: np.float32,
      G.STATS_F64: np.float64}


def run(dtypes, lo, hi, cols, n, offset=0, shape=-1):
    dev = []
    for c in cols:
        buf = torch.empty(n + 8, dtype=torch.from_numpy(c[:1]).dtype, device="cuda")
        dev.append(buf[offset:offset + n].copy_(torch.from_numpy(c)))
    with G.stats_init(G.Config(dtypes, G.STATS_EXACT, None, lo, hi)) as ctx:
        if shape >= 0:
            G.stats_set_exact_shape(ctx, shape)
        G.stats_accumulate(ctx, dev, n)
        return G.stats_raw(ctx, allow_overflow=True)


# (type, lo, hi): fields of 1..8 bytes, signed and not, odd and even byte offsets
PLANS = [
    [(G.STATS_I64, -2**62, 2**62), (G.STATS_I16, 0, 255), (G.STATS_I64, -2**62, 2**62), (G.STATS_I16, -128, 127)],
    [(G.STATS_I32, -2**31, 2**31 - 1), (G.STATS_I32, 0, 2**24 - 1), (G.STATS_I16, -2**15, 2**15 - 1),
     (G.STATS_I32, -2**23, 2**23 - 1), (G.STATS_I64, 0, 2**40 - 1), (G.STATS_I64, -2**47, 2**47 - 1),
     (G.STATS_I32, 0, 2**31 - 1), (G.STATS_I16, 0, 2**15 - 1)],
    [(G.STATS_I16, -1, 1)] * 16,
    [(G.STATS_I64, 0, 2**55), (G.STATS_I64, -2**54, 2**54), (G.STATS_I64, -2**62, 2**62),
     (G.STATS_I64, -2**62, 2**62)],
    [(G.STATS_I16, 0, 1)],
]


def values(t, lo, hi, n, rng):
    v = rng.integers(lo, hi, n, endpoint=True, dtype=np.int64)
    v[:2] = (lo, hi)[:min(2, n)]
    return v.astype(NP[t])


@pytest.mark.parametrize("n,offset,shape", [(1, 0, -1), (31, 0, -1), (961, 0, -1), (2_003, 0, -1), (2_003, 1, -1),
                                            (2_003, 0, 1), (2_003, 0, 2), (2_003, 0, 3)])
@pytest.mark.parametrize("plan", range(len(PLANS)))
def test_integer_fields(plan, n, offset, shape):
    P = PLANS[plan]
    rng = np.random.default_rng(100 * plan + n)
    cols = [values(t, lo, hi, n, rng) for t, lo, hi in P]
    raw = run([t for t, _, _ in P], [float(lo) for _, lo, _ in P], [float(hi) for _, _, hi in P], cols, n, offset, shape)
    ints = [[int(x) for x in c] for c in cols]
    assert raw.n == n
    for j, a in enumerate(ints):
        assert raw.s_exact[j] == sum(a)
        for k in range(j, len(ints)):
            exact = sum(x * y for x, y in zip(a, ints[k]))
            if -2**127 <= exact < 2**127:
                assert raw.S_exact[j][k] == exact, (j, k)


@pytest.mark.parametrize("t", [G.STATS_F32, G.STATS_F64])
@pytest.mark.parametrize("lo,hi", [(-1.0, 1.0), (0.0, 4096.0), (-1e-30, 1e-30), (0.0, 1e30)])
def test_real_fields(t, lo, hi):
    rng = np.random.default_rng(5)
    n = 1_500
    x = (lo + (hi - lo) * rng.random(n)).astype(NP[t])
    x = np.clip(x, NP[t](lo) * NP[t](0.999), NP[t](hi) * NP[t](0.999))
    x[:6] = NP[t](hi) * np.array([0.0, -0.0, 0.5, 2.0 ** -20, 2.0 ** -54, 2.0 ** -60], dtype=NP[t])
    y = rng.integers(-100, 100, n).astype(np.int16)
    raw = run([G.STATS_I16, t], [-100.0, lo], [100.0, hi], [y, x], n)
    e = np.frexp(max(abs(lo), abs(hi)))[1]
    half = Fraction(2) ** int(e) / 2 ** (55 if lo < 0 else 56)
    fx, fy = [Fraction(float(v)) for v in x], [int(v) for v in y]
    m = Fraction(2) ** int(e)

    def near(got, want, err):
        assert abs(Fraction(float(got)) - want) <= err + abs(want) / 2 ** 53

    near(raw.s[1], sum(fx), n * half)
    near(raw.S[0, 1], sum(a * b for a, b in zip(fx, fy)), 100 * n * half)
    near(raw.S[1, 1], sum(a * a for a in fx), 2 * n * half * m)
    assert raw.S_exact[0][0] == sum(b * b for b in fy)


@pytest.mark.parametrize("t,lo,hi,bad", [
    (G.STATS_I16, 0, 255, 256), (G.STATS_I16, 0, 255, -1), (G.STATS_I16, -128, 127, 128), (G.STATS_I16, -128, 127, -129),
    (G.STATS_I32, 0, 2**31 - 1, -1), (G.STATS_I32, -2**23, 2**23 - 1, 2**23), (G.STATS_I32, 0, 2**24 - 1, 2**31 - 1),
    (G.STATS_I64, 0, 2**40 - 1, 2**40), (G.STATS_I64, 0, 2**40 - 1, -1), (G.STATS_I64, -2**39, 2**39 - 1, -2**63),
    (G.STATS_F64, 0.0, 1.9, -1e-300), (G.STATS_F64, 0.0, 1.9, 2.0), (G.STATS_F64, -1.0, 1.0, 2.0),
    (G.STATS_F64, -1.0, 1.0, float("nan")), (G.STATS_F64, -1.0, 1.0, float("-inf")), (G.STATS_F32, 0.0, 1.9, float("inf"))])
def test_values_outside_their_field_are_refused(t, lo, hi, bad):
    x = np.zeros(1_000, dtype=NP[t])
    x[777] = bad
    with pytest.raises(G.StatsError) as e:
        run([G.STATS_I32, t], [0.0, float(lo)], [10.0, float(hi)], [np.ones(1_000, np.int32), x], 1_000)
    assert e.value.code == G.STATS_ERANGE
