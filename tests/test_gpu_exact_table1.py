"""The exact pass's Table 1 converter at the ends of its digit fields: every digit 0 or 255, every sign,
reals that round, vanish or are zero of either sign, values just outside; row counts around the pairs of
rows a lane takes, the 64 rows of a warp and the 960 of a stage, and past the flush of the FP32 sums.
Integers bit for bit; sums with reals within the last rounding of the exact sum of the fixed-point
values round(x 2^s), as the interface defines them."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")

COT, J = 8, 10
BOUND = {0: 2**40 - 1, 5: 65535, 9: 65535}


def config(layout):
    dt = G.stats_table1_config(layout, 1000).dtypes
    lo = [0.0] * 12
    hi = [float(BOUND.get(j, 255)) for j in range(12)]
    lo[COT], hi[COT], hi[J] = -50.0, 50.0, 9.0e5
    return G.Config(dt, G.STATS_EXACT, None, lo, hi), dt


def table(layout, n, kind):
    """Columns as numpy arrays; kind "max": all digits at their largest."""
    rng = np.random.default_rng(n)
    cfg, dt = config(layout)
    np_of = {G.STATS_I16: np.int16, G.STATS_I32: np.int32, G.STATS_I64: np.int64, G.STATS_F64: np.float64}
    cols = []
    for j in range(12):
        if j in (COT, J):
            top = np.nextafter(64.0 if j == COT else 2.0**20, 0)
            x = np.full(n, top) if kind == "max" else rng.uniform(-top if j == COT else 0.0, top, n)
            if kind != "max":
                edge = [0.0, -0.0, 5e-324, 2.0**-60, 2.0**-49, 2.0**-48, 1.5 * 2.0**-48, top]
                if j == COT:
                    edge += [-top, -64.0 + 2.0**-40, -(2.0**-49), -5e-324]
                x[:len(edge)] = edge[:n]
        else:
            b = BOUND.get(j, 255)
            x = np.full(n, b, dtype=np.int64) if kind == "max" else rng.integers(0, b, n, endpoint=True)
            if np_of[dt[j]] is np.int16:  # F and I up to the type's largest
                x = np.minimum(x, 32767)
        cols.append(np.ascontiguousarray(x.astype(np_of[dt[j]])))
    return cfg, cols


def add(ctx, cols, n, offset):
    dev = []
    for c in cols:
        buf = torch.empty(n + 8, dtype=torch.from_numpy(c[:1]).dtype, device="cuda")
        dev.append(buf[offset:offset + n].copy_(torch.from_numpy(c)))
    G.stats_accumulate(ctx, dev, n)


def fixed(x, shift):
    q = []
    for v in x:
        t = Fraction(float(v)) * 2**shift
        q.append(0 if abs(v) < 2.0**-1022 else round(t))
    return q


@pytest.mark.parametrize("layout", [G.STATS_T1_L32, G.STATS_T1_L16])
@pytest.mark.parametrize("shape,offset", [(0, 0), (0, 1), (2, 0), (3, 0)])
@pytest.mark.parametrize("n,kind", [(1, "any"), (7, "any"), (8, "max"), (63, "any"), (66, "any"), (959, "any"),
                                    (968, "max"), (1_925, "any"), (5_003, "max")])
def test_fields(layout, shape, offset, n, kind):
    cfg, cols = table(layout, n, kind)
    with G.stats_init(cfg) as ctx:
        G.stats_set_exact_shape(ctx, shape)
        G.stats_set_grid(ctx, 1)
        add(ctx, cols, n, offset)
        raw = G.stats_raw(ctx)
    shift = {COT: 54 - 6, J: 55 - 20}
    q = [fixed(c, shift[j]) if j in shift else [int(v) for v in c] for j, c in enumerate(cols)]
    assert raw.n == n
    for j in range(12):
        sj, exact = shift.get(j, 0), sum(q[j])
        if sj == 0:
            assert raw.s_exact[j] == exact
        assert abs(Fraction(float(raw.s[j])) - Fraction(exact, 2**sj)) <= Fraction(abs(exact), 2**(sj + 52))
        for k in range(j, 12):
            sk, exact = sj + shift.get(k, 0), sum(a * b for a, b in zip(q[j], q[k]))
            if sk == 0:
                assert raw.S_exact[j][k] == exact, (j, k)
            assert abs(Fraction(float(raw.S[j][k])) - Fraction(exact, 2**sk)) <= Fraction(abs(exact), 2**(sk + 52)), (j, k)


@pytest.mark.parametrize("layout", [G.STATS_T1_L32, G.STATS_T1_L16])
@pytest.mark.parametrize("row", [0, 1, 971])
def test_values_outside_are_refused(layout, row):
    n = 973
    bad = [(j, BOUND.get(j, 255) + 1) for j in range(12) if j not in (COT, J)] + [(1, -1), (0, -1)]
    bad += [(COT, 64.0), (COT, -64.0), (COT, np.inf), (COT, np.nan), (J, 2.0**20), (J, -5e-324), (J, -1.0), (J, np.nan)]
    for j, v in bad:
        cfg, cols = table(layout, n, "any")
        if v > 32767 and cols[j].dtype == np.int16:
            v = -2
        cols[j][row] = v
        for offset in (0, 1):
            with G.stats_init(cfg) as ctx:
                with pytest.raises(G.StatsError):
                    add(ctx, cols, n, offset)
                    G.stats_raw(ctx)
