"""The transposes this library is timed on, through its Python binding.

A case is one call (or one batch, or one burst of requests) on seeded synthetic
matrices of the kinds the repository's generator, tests and benchmark use.  The
inputs are drawn on the GPU with torch; plans, workspaces, output buffers, batches
and servers are made once and kept, as a program that transposes in a loop does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2012_06012_gb300 import mgt

DEV = "cuda"
TYPE_SIZES = (4, 8, 12, 16, 24, 32, 48, 64)  # byte widths of variable-width values
L2_FETCH = 32  # bytes; the L2 fetch granularity hint the benchmark sets at start-up


def _matrix(name, rows, cols, row_dist, row_mean, col_dist, len_dist, len_mean, stride, offset_bytes,
            parts=1, equal_parts=True, kind="single", **more):
    c = {"kind": kind, "rows": rows, "cols": cols, "row_dist": row_dist, "row_mean": row_mean,
         "col_dist": col_dist, "len_dist": len_dist, "len_mean": len_mean, "stride": stride,
         "offset_bytes": offset_bytes, "parts": parts, "equal_parts": equal_parts}
    if name:
        c["name"] = name
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: a thousand rows, four row blocks, 32-bit offsets (latency and launches)
        _matrix("tiny_1k", 1000, 1000, "poisson", 8.0, "uniform", "poisson1", 4.0, 8, 4, parts=4),
        # an ordinary request of the batched and serving mixes: the middle of their size range, ragged
        _matrix("member_45k", 44_721, 44_721, "lognormal", 16.0, "uniform", "geometric", 4.0, 16, 4),
        # the largest member of those mixes
        _matrix("member_2m", 1_999_993, 1_999_993, "lognormal", 16.0, "uniform", "geometric", 4.0, 16, 4),
        # the balanced multigraph: short runs of 8-byte values, 64 row blocks, 64-bit offsets
        _matrix("balanced_4m", 4_194_304, 4_194_304, "exact", 32.0, "uniform", "exact", 4.0, 8, 8, parts=64),
        # the heterogeneous multigraph (the benchmark's headline): Zipf columns, 32-byte values,
        # 256 unequal row blocks
        _matrix("heterogeneous_8m", 8_388_608, 8_388_608, "lognormal", 20.0, "zipf", "geometric", 5.0, 32, 8,
                parts=256, equal_parts=False),
        # the paper's balanced benchmark shape: 512 cells a row, ten 4-byte values a cell, 65,536 rows a
        # block; more than 2^32 values
        _matrix("paper_balanced_832k", 851_968, 851_968, "exact", 512.0, "uniform", "exact", 10.0, 4, 8, parts=13),
        # the paper's imbalanced shape: few rows of 300 thousand to 1 million cells, 128-byte values
        _matrix("long_rows", 32, 2_097_152, "uniform", 650_000.0, "uniform", "geometric", 5.0, 128, 8),
        # the way back from it (transposing twice): many rows, 48 columns of some 400 thousand cells each
        _matrix("long_columns", 1_048_575, 48, "uniform", 19.0, "uniform", "geometric", 5.0, 128, 8),
        # values of individual byte widths (one datatype per edge) on a heterogeneous matrix
        _matrix("var_width_1500k", 1_500_001, 1_500_001, "lognormal", 20.0, "zipf", "geometric", 5.0, 1, 8,
                kind="var"),
        # new values on an unchanged structure (a simulation's weights, step by step)
        _matrix("values_only_2m", 2_097_152, 2_097_152, "lognormal", 20.0, "zipf", "geometric", 5.0, 32, 8,
                kind="values"),
        # many uneven matrices in one launch of a captured graph
        {"name": "batch_24", "kind": "batch", "members": 24, "rows": 1000, "rows_hi": 2_000_000, "row_mean": 16.0,
         "len_mean": 4.0, "stride": 16},
        # a burst of requests to the serving loop: mostly small ones and one large heterogeneous one
        {"name": "serve_32", "kind": "serve", "members": 31, "rows": 1000, "rows_hi": 200_000, "row_mean": 16.0,
         "len_mean": 4.0, "stride": 16, "large_rows": 524_288},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single"] * 6 + ["var", "values", "batch", "serve"])
    if kind in ("batch", "serve"):
        c = {"kind": kind, "members": rng.randint(4, 40), "rows": _log(rng, 500, 5000),
             "rows_hi": _log(rng, 20_000, 400_000), "row_mean": round(rng.uniform(4, 24), 1),
             "len_mean": round(rng.uniform(1.5, 8), 1), "stride": rng.choice([4, 8, 16, 32])}
        if kind == "serve":
            c["large_rows"] = _log(rng, 100_000, 600_000)
        return c
    rows = _log(rng, 1000, 4_000_000)
    row_mean = round(math.exp(rng.uniform(math.log(3), math.log(200))), 1)
    row_mean = max(2.0, min(row_mean, 60e6 / rows, rows / 4))
    square = rng.random() < 0.7
    cols = rows if square else max(64, _log(rng, max(64, rows // 16), min(4_000_000, rows * 16)))
    row_mean = max(1.0, min(row_mean, cols / 4))
    len_mean = round(rng.uniform(1.5, 12), 1)
    stride = 1 if kind == "var" else rng.choice([4, 8, 12, 16, 24, 32, 64, 128])
    while rows * row_mean * len_mean * (32 if kind == "var" else stride) > 8e9:
        len_mean, row_mean = max(1.5, len_mean / 2), max(1.0, row_mean / 2)
    parts = rng.choice([1, 1, 3, 16, 100]) if square else 1
    row_dist = rng.choice(["exact", "poisson", "lognormal"])
    return _matrix(None, rows, cols, row_dist, float(int(row_mean)) if row_dist == "exact" else row_mean,
                   rng.choice(["uniform", "uniform", "zipf"]), rng.choice(["exact", "poisson1", "geometric"]),
                   len_mean, stride, rng.choice([4, 8]), parts=parts, equal_parts=rng.random() < 0.5, kind=kind)


# ------------------------------------------------------------------ inputs
def _sizes(case):
    """Cells and values of a case's matrix: the same whatever the seed."""
    C = max(1, int(round(case["rows"] * case["row_mean"])))
    per = case["len_mean"]
    return C, int(round(C * (int(per) if case["len_dist"] == "exact" else per)))


def _prefix(counts, total):
    """Offsets of runs as long as `counts` says, scaled a little so that they end at `total`."""
    p = torch.zeros(counts.numel() + 1, dtype=torch.int64, device=DEV)
    c = torch.cumsum(counts, 0)
    have = int(c[-1])
    p[1:] = c if have == total else (c.double() * (total / max(1, have))).round_().long()
    p[-1] = total
    return p


def _row_ptr(case, gen):
    R, N, mean = case["rows"], case["cols"], float(case["row_mean"])
    d = case["row_dist"]
    if d == "exact":
        n = torch.full((R,), int(mean), dtype=torch.int64, device=DEV)
    elif d == "poisson":
        n = torch.poisson(torch.full((R,), mean, device=DEV), generator=gen).long()
    elif d == "uniform":  # mean +- 54 %: rows of 300 thousand to 1 million cells for the paper's shape
        u = torch.rand(R, dtype=torch.float64, device=DEV, generator=gen)
        n = (mean * (0.4615 + 1.077 * u)).long()
    else:  # arithmetic mean `mean`, sigma 1, at most 4,096 cells a row
        z = torch.randn(R, device=DEV, generator=gen)
        n = torch.exp(z + (math.log(mean) - 0.5)).round().clamp_(max=4096).long()
    return _prefix(n.clamp_(max=max(1, N // 2)), _sizes(case)[0])


def _columns(dist, N, n, gen):
    u = torch.rand(n, dtype=torch.float64, device=DEV, generator=gen)
    if dist == "uniform":
        return (u * N).long().clamp_(max=N - 1)
    # ranks of a power law of exponent 1.1, then a multiplicative bijection rank -> column
    rank = (1.0 - u * (1.0 - (N + 1.0) ** -0.1)).pow_(-10.0).long().sub_(1).clamp_(0, N - 1)
    a = 1_000_003
    while math.gcd(a, N) != 1:
        a += 2
    return rank.mul_(a).remainder_(N)


def _structure(case, gen):
    """row_ptr, col_idx (ascending in a row, without repeats), cell_ptr; int64 / int32 / int64."""
    R, N = case["rows"], case["cols"]
    C, V = _sizes(case)
    row_ptr = _row_ptr(case, gen)
    key = torch.repeat_interleave(torch.arange(R, device=DEV) * N, row_ptr.diff())
    key += _columns(case["col_dist"], N, C, gen)
    key = torch.sort(key).values
    for again in range(12):  # repeats in a row are drawn anew, from all columns alike after a few times
        where = (key[1:] == key[:-1]).nonzero().squeeze(1) + 1
        if where.numel() == 0:
            break
        key[where] = key[where] // N * N + _columns(case["col_dist"] if again < 4 else "uniform", N, where.numel(), gen)
        key = torch.sort(key).values
    col = key.remainder_(N).int()
    del key
    mean = float(case["len_mean"])
    if case["len_dist"] == "exact":
        more = torch.full((C,), int(mean) - 1, dtype=torch.int64, device=DEV)
    elif case["len_dist"] == "poisson1":
        more = torch.poisson(torch.full((C,), mean - 1.0, device=DEV), generator=gen).long()
    else:
        u = torch.rand(C, device=DEV, generator=gen)
        more = (torch.log1p(-u) / math.log(1.0 - 1.0 / mean)).long().clamp_(0, 63)
    cell_ptr = _prefix(more, V - C)
    cell_ptr += torch.arange(C + 1, device=DEV)
    return row_ptr, col, cell_ptr


def _offsets(lens, dtype):
    p = torch.zeros(lens.numel() + 1, dtype=dtype, device=DEV)
    torch.cumsum(lens, 0, out=p[1:])
    return p


def _part_off(case, seed):
    P, R = case["parts"], case["rows"]
    if case["equal_parts"]:
        return np.array([d * R // P for d in range(P + 1)], dtype=np.int64)
    w = np.cumsum(np.exp(np.random.default_rng(seed).standard_normal(P)))
    return np.concatenate([[0], np.round(w / w[-1] * R)]).astype(np.int64)


def _payload(n_bytes, gen):
    n = (n_bytes + 7) // 8
    return torch.empty(n, dtype=torch.int64, device=DEV).random_(generator=gen).view(torch.uint8)[:n_bytes]


def _draw_matrix(case, gen, seed):
    row_ptr, col, cell_ptr = _structure(case, gen)
    odt = torch.int32 if case["offset_bytes"] == 4 else torch.int64
    row_ptr, cell_ptr, V = row_ptr.to(odt), cell_ptr.to(odt), _sizes(case)[1]
    if case["kind"] == "var":  # as many values of each width, in random order
        which = torch.randperm(V, device=DEV, generator=gen).remainder_(len(TYPE_SIZES))
        val_off = _offsets(torch.tensor(TYPE_SIZES, device=DEV)[which], torch.int64)
        del which
        return mgt.DeviceVarXCSR(case["rows"], case["cols"], case["offset_bytes"], row_ptr, col, cell_ptr,
                                 val_off, _payload(int(val_off[-1]), gen), _part_off(case, seed))
    return mgt.DeviceXCSR(case["rows"], case["cols"], case["offset_bytes"], case["stride"], row_ptr, col, cell_ptr,
                          _payload(V * case["stride"], gen), _part_off(case, seed))


def _members(case):
    """The single matrices of a batch or a burst: sizes spread over the range by their logarithm."""
    n, lo, hi = case["members"], case["rows"], case["rows_hi"]
    got = []
    for m in range(n):
        r = int(round(lo * (hi / lo) ** (m / max(1, n - 1))))
        got.append(_matrix(None, r, r, "lognormal", case["row_mean"], "uniform", "geometric", case["len_mean"],
                           case["stride"], 4))
    if case.get("large_rows"):
        r = case["large_rows"]
        got.insert(n // 2, _matrix(None, r, r, "lognormal", 20.0, "zipf", "geometric", 5.0, 32, 8))
    return got


def _inputs(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    if case["kind"] in ("batch", "serve"):
        # requests arrive in no order of size
        ms = [_draw_matrix(c, gen, seed) for c in _members(case)]
        order = np.random.default_rng(seed).permutation(len(ms))
        return [ms[i] for i in order]
    return _draw_matrix(case, gen, seed)


def _words(values):
    """The value bytes as the widest integers that divide them."""
    n = values.numel()
    return values.view(torch.int64 if n % 8 == 0 else torch.int32 if n % 4 == 0 else torch.uint8)


class _Pool:
    """Output arrays of many matrices as pieces of four buffers (256-byte aligned, gaps zero)."""

    def __init__(self, xs):
        sizes = [((x.n_cols + 1) * x.offset_bytes, x.n_cells * 4, (x.n_cells + 1) * x.offset_bytes,
                  x.n_values * x.stride) for x in xs]
        pad = [[(b + 255) // 256 * 256 for b in s] for s in sizes]
        self.buffers = [torch.zeros(sum(p[k] for p in pad), dtype=torch.uint8, device=DEV) for k in range(4)]
        at = [0, 0, 0, 0]
        self.outs = []
        for x, s, p in zip(xs, sizes, pad):
            o = [self.buffers[k][at[k]:at[k] + s[k]] for k in range(4)]
            at = [a + b for a, b in zip(at, p)]
            self.outs.append((*o, None, None))

    def whole(self):
        return [b.view(torch.int32) for b in self.buffers[:3]] + [self.buffers[3].view(torch.int64)]


def prepare(case, seed):
    mgt.l2_fetch_granularity(L2_FETCH)
    x = _inputs(case, seed)
    torch.cuda.current_stream().synchronize()
    torch.cuda.empty_cache()
    s = {"kind": case["kind"], "x": x}
    if case["kind"] in ("batch", "serve"):
        s["plans"] = [mgt.plan_for(m) for m in x]
        s["pool"] = _Pool(x)
        inps, outs = [m.arrays() for m in x], s["pool"].outs
        if case["kind"] == "batch":
            ws = mgt.alloc_workspace(mgt.batched_workspace(s["plans"]))
            s["batch"] = mgt.Batch(s["plans"], inps, outs, ws)
        else:
            s["server"] = mgt.Server(hbm_budget_bytes=60 * 10**9)
        return s
    if case["kind"] == "var":
        s["plan"] = mgt.plan_for_var(x)
        s["out"], s["out_off"] = mgt.alloc_output_var(x, parts=s["plan"].n_parts > 1)
    else:
        s["plan"] = mgt.plan_for(x)
        s["out"] = mgt.alloc_output(x, parts=s["plan"].n_parts > 1)
    s["ws"] = mgt.alloc_workspace(s["plan"].workspace_bytes)
    if case["kind"] == "values":  # the structure is transposed once; its values change afterwards
        mgt.transpose(s["plan"], x.arrays(), s["out"], s["ws"])
    return s


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["batch"].launch()
        return state["pool"].whole()
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(p, m.arrays(), o)
                   for p, m, o in zip(state["plans"], state["x"], state["pool"].outs)]
        server.drain()
        if any(server.poll(t)[:2] != (True, 0) for t in tickets):
            raise RuntimeError("a request failed")
        return state["pool"].whole()
    x, out = state["x"], state["out"]
    if kind == "var":
        mgt.transpose_var(state["plan"], x.arrays(), x.val_off, out, state["out_off"], state["ws"])
        return [*out[:3], _words(out[3]), *out[4:], state["out_off"]]
    if kind == "values":
        mgt.transpose_values(state["plan"], x.arrays(), out, state["ws"])
        return [_words(out[3])]
    mgt.transpose(state["plan"], x.arrays(), out, state["ws"])
    return [*out[:3], _words(out[3]), *out[4:]]


# -------------------------------------------------------------------- work
def _work_one(c):
    o, R, N = c["offset_bytes"], c["rows"], c["cols"]
    C, V = _sizes(c)
    if c["kind"] == "values":
        return 2 * V * c["stride"]
    payload = V * (8 + sum(TYPE_SIZES) / len(TYPE_SIZES)) if c["kind"] == "var" else V * c["stride"]
    return (R + 1) * o + (N + 1) * o + 2 * (4 * C + (C + 1) * o + payload) + \
        (16 * c["parts"] ** 2 if c["parts"] > 1 else 0)


def work(case):
    ms = _members(case) if case["kind"] in ("batch", "serve") else [case]
    return {"bytes": float(sum(_work_one(c) for c in ms)), "flops": 0.0}


# ------------------------------------------------------------------- exact
def _gather_runs(src, start, length, out):
    """out = the pieces src[start[q] : start[q] + length[q]], one after the other."""
    off = _offsets(length, torch.int64)
    C, at = start.numel(), 0
    while at < C:
        limit = off[at] + (1 << 26)
        end = max(at + 1, int(torch.searchsorted(off, limit)) - 1)
        end = min(end, C)
        a, b = int(off[at]), int(off[end])
        idx = torch.repeat_interleave(start[at:end] - off[at:end], length[at:end])
        idx += torch.arange(a, b, device=DEV)
        out[a:b] = src[idx]
        at = end
    return out


def _exact_one(x, var=False, only_values=False):
    R, N, C = x.n_rows, x.n_cols, x.n_cells
    odt = x.row_ptr.dtype
    order = torch.sort(x.col_idx, stable=True).indices
    cp = x.cell_ptr.long()
    lens = (cp[1:] - cp[:-1])[order]
    starts = cp[:-1][order]
    if var:
        a, b = x.val_off[cp[:-1]][order], x.val_off[cp[1:]][order]
        words = x.values.view(torch.int32)
        values = _gather_runs(words, a // 4, (b - a) // 4, torch.empty_like(words)).view(torch.uint8)
        widths = _gather_runs(x.val_off[1:] - x.val_off[:-1], starts, lens,
                              torch.empty(x.n_values, dtype=torch.int64, device=DEV))
        extra = [_offsets(widths, torch.int64)]
    else:
        rows_of = x.values.view(torch.int32).view(-1, x.stride // 4)
        values = _gather_runs(rows_of, starts, lens, torch.empty_like(rows_of)).view(-1).view(torch.uint8)
        extra = []
    if only_values:
        return [_words(values)]
    counts = torch.bincount(x.col_idx, minlength=N)
    row = torch.repeat_interleave(torch.arange(R, device=DEV), x.row_ptr.long().diff())
    P = len(x.part_off) - 1
    parts = [None, None]
    if P > 1:
        po = torch.from_numpy(x.part_off).to(DEV)
        key = (torch.searchsorted(po, row, right=True) - 1) * P + torch.searchsorted(po, x.col_idx.long(), right=True) - 1
        parts = [torch.bincount(key, minlength=P * P),
                 torch.zeros(P * P, dtype=torch.int64, device=DEV).index_add_(0, key, cp[1:] - cp[:-1])]
    return [_offsets(counts, odt), row[order].int(), _offsets(lens, odt), _words(values), *parts, *extra]


def exact(case, seed):
    x = _inputs(case, seed)
    if case["kind"] in ("batch", "serve"):
        pool = _Pool(x)
        for m, o in zip(x, pool.outs):
            for to, v in zip(o[:4], _exact_one(m)):
                to.copy_(v.view(torch.uint8))
        return pool.whole()
    return _exact_one(x, case["kind"] == "var", case["kind"] == "values")
