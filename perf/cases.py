"""Performance cases: the analyses that users of this library run, end to end through its public
entry points (paper_2604_23826_gb300), over the range of sizes, types and modes it serves.

A pass resets its context, adds a table's rows to it and takes the result, as a program does
that analyses one table after another with contexts it keeps:

  table1   the paper's twelve-column table, in device memory, in pinned host memory or as CSV
           text, with exact sums or with the paper's plain FP64 kernel
  ledger   integer and real columns of mixed types with declared ranges, exact sums
  tables   many independent FP32 tables in one batched call
  matrix   one FP32 table of 1..256 columns, on the tensor cores (BF16X3, BF16X4) or the FP32 cores
  stream   a growing FP64 table with a snapshot of its analysis after every chunk

Results of the FP32 modes are kept as float32, as such a program keeps them: the split modes
declare a covariance error of up to 2e-6, the pivot and the differences x - c are FP32 values, and
their FP64 digits past that would be noise.  Exact and FP64 results are kept as float64.
"""
import math
import os
import tempfile

import numpy as np
import torch

import paper_2604_23826_gb300 as G
from paper_2604_23826_gb300 import inputs

LAYOUTS = {"L32": G.STATS_T1_L32, "L16": G.STATS_T1_L16}
MODES = {"EXACT": G.STATS_EXACT, "FP64": G.STATS_FP64, "FP64_SHIFTED": G.STATS_FP64_SHIFTED,
         "BF16X3": G.STATS_BF16X3, "BF16X4": G.STATS_BF16X4, "FP32": G.STATS_FP32}
FP32_MODES = ("BF16X3", "BF16X4", "FP32")

# The ledger's columns: (storage type, lower and upper bound); the first is the record's number.
# With its ones column the exact pass carries 28 of the at most 32 digits for all eight.
LEDGER = (("int64", 1, 1e9), ("int32", 0, 65535), ("float64", 0.0, 4096.0), ("int16", -100, 100),
          ("int32", -(1 << 23), (1 << 23) - 1), ("float32", -1.0, 1.0), ("int16", 0, 6), ("int32", 0, 255))
STATS_TYPE = {"int16": G.STATS_I16, "int32": G.STATS_I32, "int64": G.STATS_I64, "float32": G.STATS_F32,
              "float64": G.STATS_F64}


def listed():
    return [
        # the parity size of the paper's table: small enough that launches, waits and the host count
        {"name": "t1_1e6", "kind": "table1", "source": "device", "layout": "L32", "mode": "EXACT", "n": 1_000_000},
        # the benchmark's table (60 GB), with the raw sums for the identifier's closed forms
        {"name": "t1_1e9", "kind": "table1", "source": "device", "layout": "L32", "mode": "EXACT", "n": 1_000_000_000},
        # the compact layout, a row count that fills no tile
        {"name": "t1_l16_ragged", "kind": "table1", "source": "device", "layout": "L16", "mode": "EXACT",
         "n": 123_456_789},
        # the paper's own kernel: FP64 on the CUDA cores, raw moments
        {"name": "t1_fp64", "kind": "table1", "source": "device", "layout": "L32", "mode": "FP64", "n": 20_000_000},
        # columns in pinned host memory, copied chunk by chunk
        {"name": "t1_host", "kind": "table1", "source": "host", "layout": "L32", "mode": "EXACT", "n": 20_000_000},
        # the paper's starting point: the table as CSV text
        {"name": "t1_csv", "kind": "table1", "source": "csv", "layout": "L32", "mode": "EXACT", "n": 1_500_000},
        # business records: integers and reals of every width but one
        {"name": "ledger_8", "kind": "ledger", "p": 8, "n": 20_000_001},
        # a wave of the many-tables workload (8..64 columns, row counts over more than three decades)
        {"name": "tables_256", "kind": "tables", "count": 256, "shapes": 3, "widths": "classes",
         "n_hi": 4_000_000, "mode": "BF16X3"},
        # the 256-column workload, as many rows as leave room for a program's other data
        {"name": "matrix_256", "kind": "matrix", "p": 256, "n": 12_000_000, "mode": "BF16X3"},
        # one 64-column table with all four split products
        {"name": "matrix_64", "kind": "matrix", "p": 64, "n": 4_000_003, "mode": "BF16X4"},
        # the most accurate FP32 mode on a width that fills no tile
        {"name": "matrix_100_fp32", "kind": "matrix", "p": 100, "n": 1_000_000, "mode": "FP32"},
        # snapshots of a growing table, each eigen-solve seeded by the one before
        {"name": "stream_48", "kind": "stream", "p": 48, "chunk": 250_001, "chunks": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["table1", "table1", "table1", "ledger", "tables", "matrix", "matrix", "stream"])
    if kind == "table1":
        source = rng.choice(["device", "device", "host", "csv"])
        mode = rng.choice(["EXACT", "EXACT", "FP64"]) if source == "device" else "EXACT"
        hi = {"device": 800_000_000 if mode == "EXACT" else 20_000_000, "host": 20_000_000, "csv": 1_500_000}[source]
        return {"kind": kind, "source": source, "layout": rng.choice(["L32", "L16"]), "mode": mode,
                "n": _log(rng, 4_000, hi)}
    if kind == "ledger":
        return {"kind": kind, "p": rng.randint(3, 8), "n": _log(rng, 4_000, 50_000_000)}
    if kind == "tables":
        return {"kind": kind, "count": _log(rng, 8, 256), "shapes": rng.randrange(1 << 20),
                "widths": rng.choice(["classes", "any"]), "n_hi": _log(rng, 10_000, 4_000_000), "mode": rng.choice(["BF16X3", "BF16X4"])}
    if kind == "matrix":
        p = _log(rng, 2, 256)
        mode = rng.choice(["BF16X3", "BF16X4", "FP32"])
        lo = max(2_000, 40 * p)
        hi = min(200_000_000, 12_000_000_000 // (4 * p)) if mode != "FP32" else min(10_000_000, 10_000_000_000 // (p * p))
        return {"kind": kind, "p": p, "n": _log(rng, lo, hi), "mode": mode}
    p = rng.randint(2, 64)
    return {"kind": kind, "p": p, "chunk": _log(rng, 4_000, 250_000), "chunks": rng.randint(2, 4)}


# ----------------------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _block(p, n, dtype=torch.float32):
    """[p, n] columns in a block whose columns start 16-byte aligned."""
    unit = 16 // (torch.finfo(dtype).bits // 8)
    return torch.empty((p, (n + unit - 1) // unit * unit), dtype=dtype, device="cuda")[:, :n]


def _correlated(p, n, seed, dtype):
    """X = Z L^T + mu with covariance eigenvalues 1 / k and means up to a thousand."""
    L, mu = inputs.wide_factor(seed, p)
    x = _block(p, n, dtype)
    if dtype == torch.float32:
        return inputs.gen_wide(torch, n, L, mu, seed, "cuda", out=x)
    g = _generator(seed)
    Lt, m = torch.as_tensor(L.T.copy(), device="cuda"), torch.as_tensor(mu, device="cuda")
    for r in range(0, n, 1 << 18):
        z = torch.randn((min(n - r, 1 << 18), p), generator=g, device="cuda", dtype=dtype)
        x[:, r:r + z.shape[0]] = torch.addmm(m, z, Lt).t()
    return x


def _ledger(p, n, seed):
    g = _generator(seed)

    def normal():
        return torch.randn(n, generator=g, device="cuda")

    def whole(lo, hi):
        return torch.randint(lo, hi + 1, (n,), generator=g, device="cuda")

    quantity = (8000.0 * torch.rand(n, generator=g, device="cuda") ** -0.5).clamp_(0, 65535).to(torch.int32)
    price = (30.0 * torch.exp(normal().double())).clamp_(0.0, 4096.0)
    score = (25.0 * normal() + 4.0 * torch.log(price).float()).round_().clamp_(-100, 100).to(torch.int16)
    balance = (1e6 * normal() + 40.0 * quantity).round_().clamp_(-(1 << 23), (1 << 23) - 1).to(torch.int32)
    rate = torch.tanh(0.3 * normal() + 0.01 * score)
    cols = [torch.arange(1, n + 1, dtype=torch.int64, device="cuda"), quantity, price, score, balance, rate,
            whole(0, 6).to(torch.int16), whole(0, 255).to(torch.int32)]
    return cols[:p]


def _table_shapes(case):
    """Rows, columns, means and spreads of each table: part of the case, the values come from the seed."""
    params = inputs.many_tables_shapes(case["shapes"], case["count"], n_hi=case["n_hi"])
    if case["widths"] == "classes":
        return params
    rng = np.random.default_rng(case["shapes"] + 1)  # any width up to 64, means and spreads as in the workload
    out = []
    for n, _, _, _ in params:
        p = int(rng.integers(1, 65))
        out.append((n, p, rng.uniform(1e3, 1e5, p), rng.uniform(0.1, 10.0, p)))
    return out


def _table1_text(cols, layout):
    """The table as CSV text without a header, on the device."""
    fd, path = tempfile.mkstemp(suffix=".csv")
    os.close(fd)
    try:
        host = [c.cpu().numpy() for c in cols]
        G.stats_csv_write(path, G.stats_table1_config(layout, len(host[0])).dtypes, len(host[0]), host)
        return torch.from_numpy(np.fromfile(path, dtype=np.uint8)).cuda()
    finally:
        os.unlink(path)


def _inputs(case, seed):
    """What the analysis reads: device columns, or tables, or chunks."""
    kind = case["kind"]
    if kind == "table1":
        return G.gen_table1(seed, case["n"], LAYOUTS[case["layout"]])
    if kind == "ledger":
        return _ledger(case["p"], case["n"], seed)
    if kind == "tables":
        tables = []
        for t, (n, p, mu, sd) in enumerate(_table_shapes(case)):
            tables.append(inputs.gen_table(torch, n, p, mu, sd, 1_000_003 * seed + t, "cuda", out=_block(p, n)))
        return tables
    if kind == "matrix":
        return _correlated(case["p"], case["n"], seed, torch.float32)
    return _correlated(case["p"], case["chunk"] * case["chunks"], seed, torch.float64)


def prepare(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    state = {"case": case, "data": data}
    if kind == "table1":
        layout, n = LAYOUTS[case["layout"]], case["n"]
        cfg = G.stats_table1_config(layout, n, MODES[case["mode"]])
        state["cols"] = data
        if case["source"] == "host":
            state["cols"] = [torch.empty(c.shape, dtype=c.dtype, pin_memory=True).copy_(c) for c in data]
            state["data"] = None
        elif case["source"] == "csv":
            state["text"] = _table1_text(data, layout)
            state["dtypes"] = cfg.dtypes
            state["cols"] = G.alloc_table1(n, layout)
            state["data"] = None
    elif kind == "ledger":
        sel = LEDGER[:case["p"]]
        cfg = G.Config([STATS_TYPE[t] for t, _, _ in sel], G.STATS_EXACT, [1] + [0] * (case["p"] - 1),
                       [lo for _, lo, _ in sel], [hi for _, _, hi in sel])
        state["cols"] = data
    elif kind == "tables":
        mode = MODES[case["mode"]]
        state["ctxs"] = [G.stats_init(G.Config([G.STATS_F32] * x.shape[0], mode)) for x in data]
        state["args"] = G.BatchArgs(state["ctxs"], [list(x) for x in data], [x.shape[1] for x in data])
        return state
    elif kind == "matrix":
        cfg = G.Config([G.STATS_F32] * case["p"], MODES[case["mode"]])
        state["cols"] = list(data)
    else:
        cfg = G.Config([G.STATS_F64] * case["p"], G.STATS_FP64_SHIFTED)
        m = case["chunk"]
        state["chunks"] = [[row[i * m:(i + 1) * m] for row in data] for i in range(case["chunks"])]
        state["stream"] = G.StreamingAnalysis(cfg)
        return state
    state["ctx"] = G.stats_init(cfg)
    return state


# ----------------------------------------------------------------------------- passes
def _outputs(an, fp32=False):
    t = np.float32 if fp32 else np.float64
    return {"mean": an.mean.astype(t, copy=False), "cov": an.cov.astype(t, copy=False),
            "corr": an.corr.astype(t, copy=False), "evals": an.evals.astype(t, copy=False),
            "evecs": an.evecs.astype(t, copy=False)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "tables":
        for c in state["ctxs"]:
            G.stats_reset(c)
        G.stats_accumulate_batched(state["args"])
        outs = G.stats_finalize_batched(state["ctxs"])
        # all tables' results one after another, as a program stores a wave
        return {f: np.concatenate([getattr(a, f).ravel() for a in outs]).astype(np.float32)
                for f in ("mean", "cov", "corr", "evals", "evecs")}
    if kind == "stream":
        s = state["stream"]
        G.stats_reset(s.ctx)
        s.prev = None  # another table: no earlier snapshot to start from
        out = []
        for chunk in state["chunks"]:
            s.update(chunk, case["chunk"])
            out.append(_outputs(s.snapshot()))
        return out
    ctx, n = state["ctx"], case.get("n")
    G.stats_reset(ctx)
    if kind == "table1" and case["source"] == "csv":
        n = G.stats_csv_parse(state["text"], state["text"].numel(), state["dtypes"], state["cols"], n)
    if kind == "table1" and case["source"] == "host":
        G.stats_accumulate_host(ctx, state["cols"], n)
    else:
        G.stats_accumulate(ctx, state["cols"], n)
    if kind == "matrix":
        return _outputs(G.stats_finalize(ctx), True)
    # mixed units: components of the correlation matrix, as in the paper's tables
    out = _outputs(G.stats_finalize(ctx, pca_on=1))
    if case["mode" if kind == "table1" else "kind"] in ("EXACT", "ledger"):
        raw = G.stats_raw(ctx)
        out |= {"n": raw.n, "s": raw.s, "S": raw.S}
    if kind == "table1" and case["source"] == "csv":
        out["columns"] = state["cols"]
    return out


# ----------------------------------------------------------------------------- work
def _columns(case):
    """(columns, bytes per row) of a one-table case."""
    kind = case["kind"]
    if kind == "table1":
        return 12, {"L32": 60, "L16": 44}[case["layout"]]
    if kind == "ledger":
        return case["p"], sum({"int16": 2, "int32": 4, "float32": 4}.get(t, 8) for t, _, _ in LEDGER[:case["p"]])
    return case["p"], (4 if kind == "matrix" else 8) * case["p"]


def _table_work(n, p, row_bytes):
    """One table read once, its results written once; the sums and the upper triangle of X^T X
    (a multiply and an add per entry), and an eigen-decomposition's ~9 p^3."""
    return n * row_bytes + 8 * (2 * p + 3 * p * p), n * p * (p + 1) + n * p + 9 * p ** 3


def work(case):
    if case["kind"] == "tables":
        each = [_table_work(n, p, 4 * p) for n, p, _, _ in _table_shapes(case)]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    p, row = _columns(case)
    n = case["n"] if "n" in case else case["chunk"] * case["chunks"]
    b, f = _table_work(n, p, row)
    if case.get("source") == "csv":
        b += 77 * n  # its text, about 77 bytes a line; the parsed columns are part of the result
    if case["kind"] == "stream":
        f += (case["chunks"] - 1) * 9 * p ** 3
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------- 64-bit results
def _moments(cols, rows=1 << 22):
    """(mean, centred cross products) of columns in 64 bits, two passes over row chunks."""
    n = cols[0].numel()
    mean = torch.stack([(c.sum(dtype=torch.float64 if c.dtype.is_floating_point else torch.int64).double() / n)
                        for c in cols])
    C = torch.zeros((len(cols), len(cols)), dtype=torch.float64, device=cols[0].device)
    rows = max(1 << 14, rows * 12 // max(12, len(cols)))
    for r in range(0, n, rows):
        X = torch.stack([c[r:r + rows].double() for c in cols]) - mean[:, None]
        C += X @ X.t()
    return n, mean.cpu().numpy(), C.cpu().numpy()


def _analysis(n, mean, C, drop=0, pca_on=0):
    mean, cov = mean[drop:], C[drop:, drop:] / (n - 1)
    sd = np.sqrt(np.diag(cov))
    corr = cov / np.outer(sd, sd)
    np.fill_diagonal(corr, 1.0)
    w, v = np.linalg.eigh(corr if pca_on else cov)
    w, v = w[::-1].copy(), v[:, ::-1].T.copy()
    big = v[np.arange(len(w)), np.argmax(np.abs(v), axis=1)]
    v *= np.where(big < 0, -1.0, 1.0)[:, None]
    return {"mean": mean, "cov": cov, "corr": corr, "evals": w, "evecs": v}


def exact(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    if kind == "tables":
        outs = [_analysis(*_moments(list(x))) for x in data]
        return {f: np.concatenate([a[f].ravel() for a in outs]) for f in ("mean", "cov", "corr", "evals", "evecs")}
    if kind == "stream":
        m = case["chunk"]
        return [_analysis(*_moments([row[:(i + 1) * m] for row in data])) for i in range(case["chunks"])]
    if kind == "matrix":
        return _analysis(*_moments(list(data)))
    cols = list(data)
    if case.get("source") == "csv":  # the text read back by numpy: its decimals rounded to the nearest double
        text = _table1_text(data, LAYOUTS[case["layout"]]).cpu().numpy()
        text[text == ord("\n")] = ord(",")
        values = np.fromstring(text[:-1].tobytes().decode(), sep=",", dtype=np.float64).reshape(-1, 12)
        cols = [torch.from_numpy(values[:, j].copy()).cuda() for j in range(12)]
    n, mean, C = _moments(cols)
    out = _analysis(n, mean, C, drop=1, pca_on=1)
    if case["mode" if kind == "table1" else "kind"] in ("EXACT", "ledger"):
        out |= {"n": n, "s": n * mean, "S": C + n * np.outer(mean, mean)}
    if case.get("source") == "csv":
        out["columns"] = [c if data[j].dtype.is_floating_point else None for j, c in enumerate(cols)]
    return out
