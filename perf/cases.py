"""The work that users of this library have it do, as measured cases.

Each listed case is one call pattern of a program that uses the library through
``paper_2609_30656_gb300.tbe``: serving lookups, training steps (forward and
de-duplicated backward, sized by the binding or into kept buffers), optimizer
steps (fused or in a second pass), the gradient of the per-sample weights, the
factorization-machine cross term, and batch replication. Sizes are those of the
repository's five workloads (``workloads.get_workload``), at full size where
three copies fit the card and with fewer tables where they do not; ``draw`` covers
the same ranges, odd sizes among them. ``exact`` states each result in float64
with plain torch.
"""

from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_2609_30656_gb300 import tbe, workloads as wl

DEV = torch.device("cuda:0")
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
INDEX = {"i32": torch.int32, "i64": torch.int64}
LR = 0.01
EPS = 1e-8

# Every key of a lookup case, with its default.
BASE = {
    "kind": "forward",      # forward | train | apply | two_pass | weight_grad | fm | replicate
    "tables": 1, "rows": 1000, "rows_lo": 0,  # rows_lo > 0: row counts log-uniform in [rows_lo, rows]
    "dims": "64",           # dims of the tables, cycling
    "dtype": "f32", "out": "f32", "index": "i64",
    "batch": 128,
    "lengths": "fixed", "mean": 4.0, "lo": 0, "hi": 0, "empty": 0.0,
    "zipf": 0.0,            # 0: uniform indices
    "weighted": False, "pooling": "sum",
    "optimizer": "",        # sgd | adagrad (apply, two_pass)
    "keep": 0.0,            # train: > 0 keeps gradient buffers for keep * n rows; 0 lets the binding size them
    "factor": 1,            # replicate
}


def _case(name, **kw):
    return {"name": name, **{**BASE, **kw}}


def listed():
    return [
        # The smallest call: one table, one small batch (the workload cfg1). Latency.
        _case("serve_one_table"),
        # A serving request over many features: a few lookups each, half-precision output.
        _case("serve_request", tables=26, rows=1_000_000, dims="64", dtype="f16", out="f16", index="i32", batch=64,
              lengths="poisson", mean=3.0, lo=0, hi=20, zipf=1.1),
        # A serving batch with ragged dims (rows that are not a power of two of 16-byte vectors).
        _case("serve_odd_dims", tables=20, rows=500_000, dims="96,48,24,80", dtype="f16", index="i32", batch=4001,
              lengths="poisson", mean=20.0, lo=0, hi=100, zipf=1.05, weighted=True, pooling="mean"),
        # A mid-size training step with fp32 tables (the workload cfg2), gradient sized by the binding.
        _case("train_fp32", kind="train", tables=8, rows=100_000, dims="128", batch=2048, lengths="poisson", mean=20.0,
              lo=0, hi=100, zipf=1.05),
        # One-hot categorical features (the workload cfg3).
        _case("train_one_hot", kind="train", tables=26, rows=10_000_000, rows_lo=10, dims="128", dtype="f16", batch=4096,
              lengths="fixed", mean=1.0, zipf=1.1),
        # Weighted mean pooling over mixed dims (the workload cfg4 at full size), gradient buffers kept.
        _case("train_weighted", kind="train", tables=64, rows=1_000_000, dims="64,128,256", dtype="bf16", batch=8192,
              lengths="lognormal", mean=50.0, lo=0, hi=500, weighted=True, pooling="mean", keep=1.0),
        # The production shape (the workload cfg5 with a fifth of its tables): skewed indices, long-tailed bags.
        _case("train_large", kind="train", tables=20, rows=5_000_000, dims="128", dtype="f16", batch=65536,
              lengths="powerlaw", mean=2.0, lo=7, hi=1000, empty=0.05, zipf=1.2, keep=0.25),
        # The same tables with uniform indices and mixed precision (no reuse of rows): bandwidth.
        _case("train_uniform_bf16", kind="train", tables=6, rows=5_000_000, dims="128", dtype="bf16", out="bf16",
              batch=65536, lengths="powerlaw", mean=2.0, lo=7, hi=1000, empty=0.05, keep=1.0),
        # A training step that ends in the tables: row-wise Adagrad fused into the backward.
        _case("train_adagrad", kind="apply", tables=16, rows=500_000, dims="64", index="i32", batch=8192,
              lengths="poisson", mean=10.0, lo=0, hi=100, zipf=1.05, optimizer="adagrad"),
        # Learned per-sample weights: their gradient.
        _case("weight_grad", kind="weight_grad", tables=24, rows=1_000_000, dims="128", dtype="f16", batch=16384,
              lengths="lognormal", mean=30.0, lo=0, hi=500, zipf=1.1),
        # The cross term over the pooled rows of 26 features, and its gradient.
        _case("fm", kind="fm", tables=26, dims="128", batch=16384),
        # A captured batch replicated to a production batch.
        _case("replicate", kind="replicate", tables=26, rows=1_000_000, batch=1024, lengths="poisson", mean=20.0, lo=0,
              hi=100, weighted=True, factor=16),
    ]


# ----------------------------------------------------------------------------- drawn cases

def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


MAX_LOOKUPS = 8_000_000
MAX_BYTES = 3 << 30   # tables, output or gradient of one drawn case


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward", "train", "train", "train", "apply", "two_pass", "weight_grad",
                       "fm", "replicate"])
    if kind == "fm":
        D = rng.choice([4, 8, 16, 20, 32, 48, 64, 96, 128, 192, 256, 512])
        T = rng.randint(2, 100)
        B = int(_log(rng, 64, 65536))
        B = max(1, min(B, MAX_BYTES // (8 * T * D)))
        return {**BASE, "kind": kind, "tables": T, "dims": str(D), "batch": B}
    c = dict(BASE, kind=kind)
    c["tables"] = T = int(_log(rng, 1, 24.99 if kind in ("apply", "two_pass") else 40.99))
    c["dtype"] = rng.choice(["f32", "f16", "bf16"])
    c["index"] = rng.choice(["i32", "i64"])
    c["out"] = rng.choice(["f32", "f32", "f16", "bf16"]) if kind != "replicate" else "f32"
    dims = ["64", "128", "32", "256", "16", "96", "48", "64,128,256", "8,24,40", "512", "80,128"]
    if c["dtype"] == "f32" and c["out"] == "f32":
        dims += ["4,12,20", "100"]
    c["dims"] = rng.choice(dims)
    mean_dim = sum(map(int, c["dims"].split(","))) / len(c["dims"].split(","))
    c["rows"] = int(_log(rng, 10, 3_000_000))
    c["rows"] = max(10, min(c["rows"], int(MAX_BYTES / (4 * mean_dim * T))))
    c["batch"] = int(_log(rng, 16, 32768))
    c["lengths"] = rng.choice(["fixed", "poisson", "lognormal", "powerlaw"])
    if c["lengths"] == "fixed":
        c["mean"] = float(int(_log(rng, 1, 40)))
    elif c["lengths"] == "powerlaw":
        c.update(mean=2.0, lo=rng.choice([1, 3, 7]), hi=1000, empty=0.05)
    else:
        c.update(mean=round(_log(rng, 1, 60), 2), hi=rng.choice([100, 500]))
    per_bag = max(_mean_length(c), 0.5)
    c["batch"] = max(1, min(c["batch"], int(MAX_LOOKUPS / (T * per_bag)), int(MAX_BYTES / (4 * mean_dim * T))))
    # the row-sparse gradient of a step has at most one row per lookup
    if kind in ("train", "two_pass"):
        c["batch"] = max(1, min(c["batch"], int(MAX_BYTES / (4 * mean_dim * T * per_bag))))
    c["zipf"] = rng.choice([0.0, 1.05, 1.1, 1.2])
    c["weighted"] = rng.random() < 0.3
    c["pooling"] = rng.choice(["sum", "sum", "mean"])
    if kind in ("apply", "two_pass"):
        c["optimizer"] = rng.choice(["sgd", "adagrad"])
    if kind == "train":
        c["keep"] = rng.choice([0.0, 1.0])
    if kind == "weight_grad":
        c["weighted"] = False
    if kind == "replicate":
        c["factor"] = rng.randint(2, 20)
        c["batch"] = max(1, c["batch"] // c["factor"])
    return c


# ----------------------------------------------------------------------------- inputs

def _workload(c):
    T = c["tables"]
    dims = [int(d) for d in c["dims"].split(",")]
    if c["rows_lo"]:
        g = np.random.RandomState(T)
        rows = [int(round(math.exp(x))) for x in g.uniform(math.log(c["rows_lo"]), math.log(c["rows"]), T)]
    else:
        rows = [c["rows"]] * T
    lengths = wl.LengthDist(c["lengths"], mean=c["mean"], lo=c["lo"], hi=c["hi"], alpha=2.0, empty_frac=c["empty"])
    return wl.Workload("perf", tuple(rows), tuple(dims[t % len(dims)] for t in range(T)), c["dtype"], c["batch"], lengths,
                       c["zipf"] or None, c["weighted"], c["pooling"] == "mean", True)


def _shuffled(x, gen):
    return x[torch.randperm(x.numel(), generator=gen, device=x.device)]


def _batch(c, w, seed):
    """A jagged batch. Each table's bag lengths and its lookups' ranks are drawn from
    the case alone, so that every seed has as many lookups and distinct rows (results
    of one size); the seed says in which order they come and which row has which rank."""
    fixed = torch.Generator(device=DEV).manual_seed(w.num_tables * 1_000_003 + w.batch)
    own = torch.Generator(device=DEV).manual_seed(seed)
    lengths, indices = [], []
    for rows in w.rows:
        lens = _shuffled(wl.bag_lengths(w, fixed, w.batch, DEV), own)
        n = int(lens.sum())
        if w.zipf_alpha is None:
            ranks = torch.randint(0, rows, (n,), generator=fixed, device=DEV)
        else:
            ranks = wl.zipf_ranks(rows, w.zipf_alpha, n, fixed, DEV)
        row_of = torch.randperm(rows, generator=own, device=DEV)
        lengths.append(lens)
        indices.append(row_of[_shuffled(ranks, own)])
    offsets = torch.zeros(w.num_tables * w.batch + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.cat(lengths), 0, out=offsets[1:])
    indices = torch.cat(indices)
    weights = torch.rand(indices.numel(), generator=own, device=DEV) if w.weighted else None
    return indices.to(INDEX[c["index"]]), offsets.to(INDEX[c["index"]]), weights


class _State:
    """What a program holds before the call: batch, tables, handle, kept buffers."""


def _inputs(c, seed):
    s = _State()
    s.case = c
    if c["kind"] == "fm":
        D = int(c["dims"])
        g = torch.Generator(device=DEV).manual_seed(seed)
        s.y = torch.randn(c["batch"], c["tables"] * D, generator=g, device=DEV) * 0.1
        s.grad_fm = torch.randn(c["batch"], generator=g, device=DEV)
        return s
    s.w = w = _workload(c)
    s.indices, s.offsets, s.weights = _batch(c, w, seed)
    s.n = int(s.indices.numel())
    if c["kind"] == "replicate":
        return s
    s.tables = wl.make_tables(w, seed, DEV)
    if c["kind"] != "forward":
        s.grad_out = wl.make_grad_out(w, seed, DEV).to(DTYPES[c["out"]])
    if c["optimizer"] == "adagrad":
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        # a table some way into training: no row's state is zero
        s.state = [torch.rand(t.shape[0], generator=g, device=DEV) + 0.1 for t in s.tables]
    else:
        s.state = None
    return s


def _kept_room(s):
    """(rows, values) of gradient buffers with room for `keep` of each table's lookups."""
    w = s.w
    starts = s.offsets[::w.batch].tolist()
    rows = [min(int(s.case["keep"] * (b - a)) + 64, r) for a, b, r in zip(starts, starts[1:], w.rows)]
    return sum(rows), sum(r * d for r, d in zip(rows, w.dims))


def prepare(case, seed):
    c = case
    s = _inputs(c, seed)
    if c["kind"] in ("fm", "replicate"):
        return s
    s.m = tbe.TBE(s.tables, pooling=c["pooling"], index_dtype=INDEX[c["index"]], out_dtype=DTYPES[c["out"]])
    s.m.reserve(c["batch"], s.n)
    if c["kind"] == "train" and c["keep"]:
        s.g = s.m.alloc_grad(*_kept_room(s))
        for t in (s.g.unique_ids, s.g.grad_offsets, s.g.grads):
            t.zero_()  # so that the room that a batch does not fill is the same in every run
    return s


# ----------------------------------------------------------------------------- one pass

def _grad(g):
    return {"unique_ids": g.unique_ids, "table_offsets": g.table_offsets, "grad_offsets": g.grad_offsets,
            "grads": g.grads, "num_unique": g.num_unique_dev, "num_floats": g.num_floats_dev}


def run(state):
    s, c = state, state.case
    kind = c["kind"]
    if kind == "fm":
        return {"fm": tbe.fm_forward(s.y, c["tables"]), "grad_y": tbe.fm_backward(s.y, s.grad_fm, c["tables"])}
    if kind == "replicate":
        ind, off, w = tbe.replicate_batch(s.indices, s.offsets, s.weights, c["tables"], c["factor"])
        return {"indices": ind, "offsets": off, "weights": w}
    if kind == "weight_grad":
        return {"grad_weights": s.m.weight_grad(s.indices, s.offsets, s.grad_out)}
    y = s.m.forward(s.indices, s.offsets, s.weights)
    if kind == "forward":
        return {"y": y}
    if kind == "train":
        if c["keep"]:
            g = s.m.backward_into(s.g, s.indices, s.offsets, s.grad_out, s.weights)
        else:
            g = s.m.backward(s.indices, s.offsets, s.grad_out, s.weights)
        return {"y": y, **_grad(g)}
    if kind == "apply":
        s.m.backward_apply(s.indices, s.offsets, s.grad_out, s.weights, optimizer=c["optimizer"], lr=LR, eps=EPS,
                           state=s.state)
        return {"y": y, "tables": s.tables, "state": s.state}
    g = s.m.backward(s.indices, s.offsets, s.grad_out, s.weights)
    s.m.apply_sparse(g, optimizer=c["optimizer"], lr=LR, eps=EPS, state=s.state)
    return {"y": y, **_grad(g), "tables": s.tables, "state": s.state}


# ----------------------------------------------------------------------------- float64

_SLAB = 1 << 28  # float64 values gathered at once


def _per_table(s):
    """(table, its lookups' rows, bags, coefficients) in float64 per table."""
    w, B = s.w, s.w.batch
    starts = s.offsets[::B].tolist()
    for t in range(w.num_tables):
        lo, hi = starts[t], starts[t + 1]
        off = s.offsets[t * B:(t + 1) * B + 1].long()
        lens = off[1:] - off[:-1]
        bag = torch.repeat_interleave(torch.arange(B, device=DEV), lens, output_size=hi - lo)
        coef = torch.ones(hi - lo, dtype=torch.float64, device=DEV) if s.weights is None else s.weights[lo:hi].double()
        if w.mean:
            coef = coef / lens.double()[bag]
        yield t, s.indices[lo:hi].long(), bag, coef


def _slabs(n, dim):
    step = max(1, _SLAB // dim)
    return [(i, min(i + step, n)) for i in range(0, n, step)]


def exact(case, seed):
    c = case
    s = _inputs(c, seed)
    if c["kind"] == "fm":
        v = s.y.double().view(c["batch"], c["tables"], -1)
        S = v.sum(1)
        grad = s.grad_fm.double()[:, None, None] * (S[:, None, :] - v)
        return {"fm": 0.5 * (S.square() - v.square().sum(1)).sum(1), "grad_y": grad.view(c["batch"], -1)}
    if c["kind"] == "replicate":
        if s.weights is None:
            return None  # whole numbers only
        starts = s.offsets[::c["batch"]].tolist()
        parts = [s.weights[a:b].double().repeat(c["factor"]) for a, b in zip(starts, starts[1:])]
        return {"indices": None, "offsets": None, "weights": torch.cat(parts)}
    w, B = s.w, s.w.batch
    y = torch.zeros(B, w.sum_dims, dtype=torch.float64, device=DEV)
    if c["kind"] == "weight_grad":
        gw = torch.empty(s.n, dtype=torch.float64, device=DEV)
    grads, col, pos, ids = [], 0, 0, 0
    for t, rows, bag, coef in _per_table(s):
        d = w.dims[t]
        n = rows.numel()
        if c["kind"] == "weight_grad":
            go = s.grad_out[:, col:col + d]
            for i, j in _slabs(n, d):
                dots = (go[bag[i:j]].double() * s.tables[t][rows[i:j]].double()).sum(1)
                gw[pos + i:pos + j] = dots * coef[i:j]
        else:
            out = torch.zeros(B, d, dtype=torch.float64, device=DEV)
            for i, j in _slabs(n, d):
                out.index_add_(0, bag[i:j], s.tables[t][rows[i:j]].double() * coef[i:j, None])
            y[:, col:col + d] = out
        if c["kind"] in ("train", "apply", "two_pass"):
            uniq, inv = torch.unique(rows, return_inverse=True)
            G = torch.zeros(uniq.numel(), d, dtype=torch.float64, device=DEV)
            go = s.grad_out[:, col:col + d]
            for i, j in _slabs(n, d):
                G.index_add_(0, inv[i:j], go[bag[i:j]].double() * coef[i:j, None])
            ids += uniq.numel()
            if c["kind"] != "apply":
                grads.append(G.reshape(-1))
            if c["optimizer"]:
                scale = LR
                if s.state is not None:
                    m = s.state[t].double()
                    m[uniq] += G.square().mean(1)
                    s.state[t] = m
                    scale = LR / (m[uniq].sqrt() + EPS)[:, None]
                E = s.tables[t].double()
                E[uniq] -= scale * G
                s.tables[t] = E
        col += d
        pos += n
    if c["kind"] == "weight_grad":
        return {"grad_weights": gw}
    res = {"y": y}
    if c["kind"] in ("train", "two_pass"):
        flat = torch.cat(grads)
        if c["keep"]:
            whole = torch.zeros(_kept_room(s)[1], dtype=torch.float64, device=DEV)
            whole[:flat.numel()] = flat
            flat = whole
        elif flat.numel() < 4:
            flat = None
        res.update(unique_ids=None, table_offsets=None, grad_offsets=None, grads=flat, num_unique=None, num_floats=None)
    if c["optimizer"]:
        res.update(tables=s.tables, state=s.state)
    return res


# ----------------------------------------------------------------------------- work, tolerance

@lru_cache(maxsize=None)
def _mean_of_lengths(kind, mean, lo, hi, empty):
    if kind == "lognormal":
        z = np.linspace(-8, 8, 20001)
        p = np.exp(-0.5 * z * z)
        x = np.clip(np.round(np.exp(math.log(mean) - 0.5 + z)), lo, hi)
        return float((x * p).sum() / p.sum())
    if kind == "powerlaw":
        k = np.arange(lo, hi + 1, dtype=np.float64)
        return float((1 - empty) * (1 / k).sum() / (1 / (k * k)).sum())
    return mean


def _mean_length(c):
    return _mean_of_lengths(c["lengths"], c["mean"], c["lo"], c["hi"], c["empty"])


@lru_cache(maxsize=None)
def _touched(rows, n, zipf):
    """Expected distinct rows among n lookups."""
    if zipf:
        p = np.arange(1, rows + 1, dtype=np.float64) ** -zipf
        p /= p.sum()
        return float(-np.expm1(-n * p).sum())
    return rows * -math.expm1(-n / rows)


def work(case):
    c = case
    if c["kind"] == "fm":
        size = c["batch"] * c["tables"] * int(c["dims"])
        # y once, its gradient, the two vectors; sums, squares and the gradient's two operations
        return {"bytes": 8 * size + 8 * c["batch"], "flops": 5 * size}
    w = _workload(c)
    per_table = int(_mean_length(c) * c["batch"])
    n = per_table * c["tables"]
    eb = 4 if c["dtype"] == "f32" else 2
    ob = 4 if c["out"] == "f32" else 2
    ib = 4 if c["index"] == "i32" else 8
    batch_in = n * (ib + (4 if c["weighted"] else 0)) + ib * (c["tables"] * c["batch"] + 1)
    if c["kind"] == "replicate":
        return {"bytes": (1 + c["factor"]) * batch_in, "flops": 0}
    touched = [_touched(r, per_table, c["zipf"]) for r in w.rows]
    rows = sum(u * d for u, d in zip(touched, w.dims))  # values of the touched rows
    values = per_table * sum(w.dims)                    # values of every lookup's row
    slab = c["batch"] * w.sum_dims * ob                 # the pooled output, or its gradient
    per = 2 if c["weighted"] else 1
    if c["kind"] == "weight_grad":
        return {"bytes": batch_in + rows * eb + slab + 4 * n, "flops": 2 * values}
    total, flops = batch_in + rows * eb + slab, per * values
    if c["kind"] == "forward":
        return {"bytes": total, "flops": flops}
    total, flops = total + slab, 2 * flops
    if c["kind"] in ("train", "two_pass"):
        total += rows * 4 + 16 * sum(touched)
    if c["optimizer"]:
        total += rows * eb + (8 * sum(touched) if c["optimizer"] == "adagrad" else 0)
        flops += 2 * rows
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """Measured against exact(): 32-bit sums are 4e-8 to 2.3e-7 off (2-norm), results
    rounded to fp16 2.1e-4 to 2.3e-4, to bf16 1.7e-3; about four times that, and for
    single values of the narrow types two of their units."""
    c = case
    if c["kind"] == "replicate":
        return "exact"
    if c["kind"] not in ("fm", "weight_grad"):
        stored = {c["out"]} | ({c["dtype"]} if c["optimizer"] else set())
        if "bf16" in stored:
            return {"rel": 6e-3, "max": 1.6e-2}
        if "f16" in stored:
            return {"rel": 8e-4, "max": 2e-3}
    return {"rel": 1e-6, "max": 4e-5}
