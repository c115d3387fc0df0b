"""CSV fields taken eight characters at a time, at the lengths and alignments where that can go wrong.

Reals: the same number is written plainly and with an exponent of zero, which the character loop
reads; both must give the same bits, in FP64 also those of Python's correctly rounded float().
Integers against int().  The text starts at every offset from a 16-byte boundary, ends with and
without a newline, with and without carriage returns."""
import random

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
G = pytest.importorskip("paper_2604_23826_gb300")

TORCH = {G.STATS_I16: torch.int16, G.STATS_I32: torch.int32, G.STATS_I64: torch.int64, G.STATS_F32: torch.float32,
         G.STATS_F64: torch.float64}


def parse(text, dtypes, rows, offset=0):
    buf = torch.zeros(len(text) + 64, dtype=torch.uint8, device="cuda")
    d = buf[offset:offset + len(text)]
    d.copy_(torch.frombuffer(bytearray(text), dtype=torch.uint8))
    cols = [torch.zeros(rows, dtype=TORCH[t], device="cuda") for t in dtypes]
    assert G.stats_csv_parse(d, len(text), dtypes, cols, rows) == rows
    return [c.cpu().numpy() for c in cols]


def reals(rng, n):
    out = ["0", "-0", "0.0", "-0.000", "5.", "1", "9007199254740993", "0.1", "00012.50", "1.0000000000000000",
           "0.0088516559960109401", "123456789012345678.9", "1234567890123456789", "0.1234567890123456789",
           "9999999999999999999", "00000000000000000000000012.5", "3.4028234", "8388609.5"]
    while len(out) < n:
        a, b = rng.randint(1, 19), rng.randint(0, 19)
        s = "".join(rng.choice("0123456789") for _ in range(a))
        if rng.random() < 0.8:
            s += "." + "".join(rng.choice("0123456789") for _ in range(b))
        if len(s.replace(".", "").lstrip("0")) <= 19:  # the digits that count; the rest is refused
            out.append(rng.choice(["", "-", "+"]) + s)
    return out


@pytest.mark.parametrize("t", [G.STATS_F64, G.STATS_F32])
@pytest.mark.parametrize("offset,newline,last", [(0, "\n", True), (1, "\n", False), (7, "\r\n", True), (8, "\n", False),
                                                (13, "\r\n", False)])
def test_plain_reals_equal_the_character_loop(t, offset, newline, last):
    xs = reals(random.Random(offset), 3_000)
    text = newline.join(f"{x},{x}e0,{x}" for x in xs) + (newline if last else "")
    a, b, c = parse(text.encode(), [t, t, t], len(xs), offset)
    u = np.uint64 if t == G.STATS_F64 else np.uint32
    assert np.array_equal(a.view(u), b.view(u)) and np.array_equal(c.view(u), b.view(u))
    if t == G.STATS_F64:
        assert np.array_equal(a.view(u), np.array([float(x) for x in xs]).view(u))


@pytest.mark.parametrize("t,hi", [(G.STATS_I16, 2**15), (G.STATS_I32, 2**31), (G.STATS_I64, 2**63)])
@pytest.mark.parametrize("offset", [0, 3, 11])
def test_integers_of_every_length(t, hi, offset):
    rng = random.Random(hi + offset)
    vals = [0, hi - 1, -hi, 1, -1] + [rng.choice([1, -1]) * (rng.randrange(min(hi, 10 ** d))) for d in range(1, 20) for _ in range(40)]
    xs = [("+" if v >= 0 and rng.random() < 0.1 else "-" if v < 0 else "") +
          "0" * (rng.randrange(3) if len(str(abs(v))) < 17 else 0) + str(abs(v)) for v in vals]
    text = "\n".join(f"{x},{x}" for x in xs)
    a, b = parse(text.encode(), [t, t], len(xs), offset)
    assert a.tolist() == vals and b.tolist() == vals


@pytest.mark.parametrize("field,t,code", [
    ("", G.STATS_I32, "EFORMAT"), ("-", G.STATS_I32, "EFORMAT"), ("12a", G.STATS_I32, "EFORMAT"), ("1.5", G.STATS_I32, "EFORMAT"),
    ("12345678 ", G.STATS_I32, "EFORMAT"), ("2147483648", G.STATS_I32, "ERANGE"), ("-32769", G.STATS_I16, "ERANGE"),
    ("9223372036854775808", G.STATS_I64, "ERANGE"), ("12345678901234567890", G.STATS_I64, "EFORMAT"),
    (".", G.STATS_F64, "EFORMAT"), ("1.2.3", G.STATS_F64, "EFORMAT"), ("1.5x", G.STATS_F64, "EFORMAT"),
    ("1.23456789012345678912", G.STATS_F64, "EFORMAT"), ("nan", G.STATS_F64, "EFORMAT"), ("1e", G.STATS_F64, "EFORMAT")])
def test_what_was_refused_stays_refused(field, t, code):
    text = "\n".join(["7,7"] * 50 + [f"{field},7"] + ["7,7"] * 50 + [f"7,{field}"])
    with pytest.raises(G.StatsError) as e:
        parse(text.encode(), [t, t], 102)
    assert e.value.code == getattr(G, "STATS_" + code) and e.value.bad_line == 50


def test_lines_across_tiles():
    """Empty-field-free lines of 2 to 9000 characters: newlines at every place of the 4 KB tiles."""
    rng = random.Random(3)
    vals = [rng.randrange(10 ** rng.randint(1, 15)) for _ in range(6_000)]
    text = "\n".join(str(v) + "," + "9" * rng.choice([1, 1, 2, 30, 500] + [9000] * (i % 500 == 0)) for i, v in enumerate(vals))
    (a,) = parse(text.encode(), [G.STATS_I64], len(vals), 5)
    assert a.tolist() == vals
