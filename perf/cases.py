"""Performance cases of the aggregation library.

Each case is one call (or one run of a kept plan) through the Python binding of
the C ABI, on columns that are already in device memory, over the sizes, key
distributions, value types and functions the library is used with. Results are
read where the library leaves them: in the device arrays of the result struct.

  listed()             the cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  columns, plan and options of one call, from the seed
  run(state)           the call; its outputs
  work(case)           the bytes a call cannot do without
  exact(case, seed)    the float outputs in float64, from plain torch
"""
from __future__ import annotations

import ctypes
import functools
import math

import numpy as np
import torch

import paper_2606_10030_gb300 as agg

SUM, MIN, MAX, COUNT, AVG = "sum", "min", "max", "count", "avg"
BITS = {SUM: agg.AGG_SUM, MIN: agg.AGG_MIN, MAX: agg.AGG_MAX, COUNT: agg.AGG_COUNT, AVG: agg.AGG_AVG}
ALL = "sum,min,max,count,avg"
SIZE = {"i32": 4, "u32": 4, "f32": 4, "i64": 8, "f64": 8}
FLOATS = ("f32", "f64")
CHUNK = 1 << 25  # rows made at a time
BATCH_QUERIES = 12


def listed():
    return [
        # A small column's summary: the call's own latency counts.
        {"name": "scan_i32_1m", "path": "scan", "rows": 1 << 20, "dtype": "i32", "ops": ALL},
        # The summary of a large float64 column (odd length).
        {"name": "scan_f64_100m", "path": "scan", "rows": 100_000_007, "dtype": "f64", "ops": ALL},
        # A bit-packed integer column, decoded inside the scan.
        {"name": "packed_i32_32m", "path": "packed", "rows": (1 << 25) + 11, "dtype": "i32", "ops": ALL},
        # A report over a small table: a few dozen groups, launches and read-backs count.
        {"name": "groupby_f64_50k", "path": "groupby", "rows": 50_021, "keys": 100, "skew": 0.0, "dtype": "f64",
         "ops": ALL, "strategy": "auto"},
        # An ordinary query: a few million rows, skewed keys, more groups than one shared table holds.
        {"name": "groupby_i32_3m", "path": "groupby", "rows": 3_000_017, "keys": 10_000, "skew": 1.0, "dtype": "i32",
         "ops": "sum,count,min,max", "strategy": "auto"},
        # Few groups over many rows (the benchmark's low-cardinality GROUP BY).
        {"name": "groupby_i64_64m", "path": "groupby", "rows": 1 << 26, "keys": 1024, "skew": 0.0, "dtype": "i64",
         "ops": "sum,count,min,max", "strategy": "auto"},
        # Many groups of float64 values, every function.
        {"name": "groupby_f64_16m", "path": "groupby", "rows": 16_000_057, "keys": 1 << 20, "skew": 0.0, "dtype": "f64",
         "ops": ALL, "strategy": "auto"},
        # Nearly distinct keys: as many groups as rows, within a factor of two.
        {"name": "groupby_u32_2m_wide", "path": "groupby", "rows": 2_000_003, "keys": 1_500_000, "skew": 0.0,
         "dtype": "u32", "ops": "sum,count", "strategy": "auto"},
        # High cardinality under skew (the benchmark's 2^28-row float32 column, 14 M groups).
        {"name": "groupby_f32_256m", "path": "groupby", "rows": 1 << 28, "keys": 1 << 24, "skew": 1.0, "dtype": "f32",
         "ops": "sum,avg", "strategy": "auto"},
        # The headline table: 2^30 rows, Zipf(1.0) over 2^16 keys, int64, the learned selector's plan.
        {"name": "table_i64_1g", "path": "groupby", "rows": 1 << 30, "keys": 1 << 16, "skew": 1.0, "dtype": "i64",
         "ops": ALL, "strategy": "learned"},
        # Deterministic float sums (exactly rounded), the reproducible-report option.
        {"name": "exact_f32_32m", "path": "exact", "rows": (1 << 25) + 33, "keys": 4096, "skew": 0.8, "dtype": "f32",
         "ops": "sum,count,avg", "strategy": "auto"},
        # A dashboard's queries in one kept plan: uneven sizes and types, replayed.
        {"name": "batch_12", "path": "batch", "low": 1 << 14, "rows": 1 << 23, "keys": 1 << 18, "ops": "sum,count,min,max"},
    ]


def _between(rng, lo, hi):
    """An integer of [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    path = rng.choice(["scan", "scan", "packed", "groupby", "groupby", "groupby", "groupby", "groupby", "exact", "batch"])
    ops = rng.choice([ALL, "sum,count,min,max", "sum,count", "sum,avg", "sum,count,avg", "min,max"])
    if path == "scan":
        return {"path": path, "rows": _between(rng, 1 << 20, 1 << 28), "dtype": rng.choice(list(SIZE)), "ops": ops}
    if path == "packed":
        return {"path": path, "rows": _between(rng, 1 << 20, 1 << 25), "dtype": rng.choice(["i32", "u32", "i64"]), "ops": ops}
    if path == "batch":
        rows = _between(rng, 1 << 17, 1 << 23)
        return {"path": path, "low": 1 << 14, "rows": rows, "keys": _between(rng, 64, 1 << 18), "ops": "sum,count,min,max"}
    skew = rng.choice([0.0, 0.0, round(rng.uniform(0.5, 1.5), 3)])
    if path == "exact":
        rows = _between(rng, 1 << 18, 1 << 25)
        return {"path": path, "rows": rows, "keys": _between(rng, 1, min(rows, 1 << 20)), "skew": skew,
                "dtype": rng.choice(FLOATS), "ops": "sum,count,avg", "strategy": "auto"}
    rows = _between(rng, 20_000, 1 << 28)
    return {"path": path, "rows": rows, "keys": _between(rng, 1, min(rows, 1 << 24)), "skew": skew,
            "dtype": rng.choice(list(SIZE)), "ops": ops, "strategy": rng.choice(["auto", "auto", "learned"])}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + stream) & 0x7FFFFFFFFFFF)
    return g


def _values(dtype, n, seed, stream=1):
    """i32 uniform in [-2^20, 2^20); i64 and u32 uniform in [0, 2^32); floats N(0, 1) x 1e3."""
    g = _generator(seed, stream)
    d = torch.device("cuda")
    if dtype == "i32":
        return torch.randint(-(1 << 20), 1 << 20, (n,), dtype=torch.int32, generator=g, device=d)
    if dtype == "i64":
        return torch.randint(0, 1 << 32, (n,), dtype=torch.int64, generator=g, device=d)
    if dtype == "u32":
        return torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int32, generator=g, device=d).view(torch.uint32)
    return torch.randn(n, dtype=torch.float32 if dtype == "f32" else torch.float64, generator=g, device=d).mul_(1e3)


def _domain(rank, seed):
    """Distinct 32-bit keys for ranks: a bijective mixer (Wellons' lowbias32) of the salted rank, as int64."""
    m = 0xFFFFFFFF
    x = rank ^ ((int(seed) * 0x9E3779B1 + 0x7F4A7C15) & m)
    x = ((x ^ (x >> 16)) * 0x7FEB352D) & m
    x = ((x ^ (x >> 15)) * 0x846CA68B) & m
    return x ^ (x >> 16)


@functools.lru_cache(maxsize=1)
def _cdf(count, skew):
    """Zipf(skew) over ranks 1..count (summed in a fixed order, so that every run draws the same ranks)."""
    c = np.cumsum(np.arange(1, count + 1, dtype=np.float64) ** -float(skew))
    return torch.from_numpy(c / c[-1]).to("cuda")


def _keys(n, count, skew, seed, stream=2):
    """uint32 keys: ranks uniform or Zipf(skew) over `count` distinct random keys. The ranks drawn are
    the same for every seed (so that every seed has as many groups), the keys that stand for them and
    the row they begin at are the seed's."""
    g = _generator(12345, stream)
    out = torch.empty(n, dtype=torch.int32, device="cuda")
    cdf = _cdf(count, skew) if skew > 0 else None
    for a in range(0, n, CHUNK):
        u = torch.rand(min(CHUNK, n - a), dtype=torch.float64, generator=g, device="cuda")
        rank = torch.searchsorted(cdf, u, right=True) if cdf is not None else (u * count).long()
        k = _domain(rank.clamp_(max=count - 1), seed)
        out[a: a + k.numel()] = k.to(torch.int32)  # the low 32 bits
    return torch.roll(out, int(seed) * 7_368_787 % n).view(torch.uint32)


def _ops(case):
    names = case["ops"].split(",")
    return names, sum(BITS[x] for x in names)


def _queries(case, seed):
    """The batch's queries: rows and keys spread over their range, every value type, uniform and skewed keys."""
    out = []
    for j in range(BATCH_QUERIES):
        f = j / (BATCH_QUERIES - 1)
        n = int(round(case["low"] * (case["rows"] / case["low"]) ** f)) | 1
        count = max(1, min(n, int(round(case["keys"] ** (((5 * j) % BATCH_QUERIES) / (BATCH_QUERIES - 1))))))
        dtype = ["i32", "i64", "f32", "f64"][j % 4]
        skew = [0.0, 1.0, 0.7][j % 3]
        out.append((dtype, _keys(n, count, skew, seed + 7919 * j), _values(dtype, n, seed + 7919 * j)))
    return out


def _strategy(case):
    if case["strategy"] == "learned":
        from paper_2606_10030_gb300 import selector
        if selector.install_default():
            return agg.AGG_STRAT_LEARNED
    return agg.AGG_STRAT_AUTO


def prepare(case, seed):
    names, ops = _ops(case)
    s = {"path": case["path"], "names": names, "ops": ops}
    if case["path"] == "scan":
        s["dtype"] = case["dtype"]
        s["col"] = _values(case["dtype"], case["rows"], seed)
        s["out"], s["fields"] = _scalar(names, case["dtype"] in FLOATS)
    elif case["path"] == "packed":
        s["dtype"] = case["dtype"]
        s["col"] = agg.agg_pack_for(_packable(case, seed).cpu()).to("cuda")
        s["out"], s["fields"] = _scalar(names, False)
    elif case["path"] == "batch":
        s["queries"] = _queries(case, seed)
        s["dtypes"] = [q[0] for q in s["queries"]]
        s["plan"] = agg.BatchPlan([(k, v, ops, agg.AGG_STRAT_AUTO) for _, k, v in s["queries"]])
    else:
        s["dtype"] = case["dtype"]
        s["keys"] = _keys(case["rows"], case["keys"], case["skew"], seed)
        s["vals"] = _values(case["dtype"], case["rows"], seed)
        s["opts"] = agg.options(_strategy(case), flags=agg.AGG_FLAG_EXACT_SUM if case["path"] == "exact" else 0)
    return s


def _packable(case, seed):
    """A column whose neighbours are near each other (a slowly drifting measure), so that its frames pack."""
    v = _values(case["dtype"], case["rows"], seed)
    drift = torch.arange(case["rows"], device="cuda", dtype=torch.int64) >> 6
    if case["dtype"] == "i32":
        return ((v >> 4) + drift.to(torch.int32)).contiguous()
    if case["dtype"] == "u32":
        return ((v.view(torch.int32).to(torch.int64) & 0xFFFF) + drift).to(torch.int32).view(torch.uint32)
    return (v >> 12) + (drift << 8)


# ---------------------------------------------------------------------------
# The call
# ---------------------------------------------------------------------------
class _Array:
    """A device array of a result struct, for torch to read in place (it keeps the result alive)."""
    __slots__ = ("__cuda_array_interface__", "owner")

    def __init__(self, owner, ptr, n, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": typestr, "data": (ptr or 0, False), "version": 2}


def _arrays(groups, names, fp):
    """Keys and the requested functions of a result, in device memory."""
    g = ctypes.cast(groups._ptr, ctypes.POINTER(agg.AggGroups)).contents
    n = groups.num_groups
    t = "<f8" if fp else "<i8"
    out = {"keys": torch.as_tensor(_Array(groups, g.keys, n, "<i4"), device="cuda")}
    if COUNT in names:
        out[COUNT] = torch.as_tensor(_Array(groups, g.count, n, "<i8"), device="cuda")
    for name, ptr, kind in ((SUM, g.sum, t), (MIN, g.min, t), (MAX, g.max, t), (AVG, g.avg, "<f8")):
        if name in names:
            out[name] = torch.as_tensor(_Array(groups, ptr, n, kind), device="cuda")
    return out


def _scalar(names, fp):
    """A device agg_scalar and its requested fields. (err_bound is left out: it depends on how the
    scan is cut into threads, and any value that bounds the error is right.)"""
    out = torch.empty(agg.SCALAR_BYTES, dtype=torch.uint8, device="cuda")
    i, f = out[:64].view(torch.int64), out[:64].view(torch.float64)
    got = {COUNT: i[0], SUM: f[2] if fp else i[1], AVG: f[3], MIN: f[6] if fp else i[4], MAX: f[7] if fp else i[5]}
    return out, {k: got[k] for k in names}


def run(state):
    names, ops = state["names"], state["ops"]
    if state["path"] == "scan":
        agg.agg_reduce(state["col"], ops, out=state["out"])
        return state["fields"]
    if state["path"] == "packed":
        agg.agg_reduce_packed(state["col"], ops, out=state["out"])
        return state["fields"]
    if state["path"] == "batch":
        plan = state["plan"]
        plan.run()
        return [_arrays(plan.result(i), names, d in FLOATS) for i, d in enumerate(state["dtypes"])]
    g = agg.agg_groupby(state["keys"], state["vals"], ops, state["opts"])
    return _arrays(g, names, state["dtype"] in FLOATS)


# ---------------------------------------------------------------------------
# What a call cannot do without
# ---------------------------------------------------------------------------
def _groups(n, count, skew):
    """Expected distinct keys among n draws (ranks on a logarithmic grid where there are many)."""
    if skew == 0:
        return -count * math.expm1(n * math.log1p(-1.0 / count)) if count > 1 else 1.0
    edges = np.unique(np.round(np.exp(np.linspace(0.0, math.log(count + 1.0), 4096)))) if count > 4096 else np.arange(1.0, count + 2)
    mid, width = (edges[:-1] + edges[1:] - 1) / 2, np.diff(edges)
    p = mid ** -skew
    p /= float((p * width).sum())
    return float((-np.expm1(-n * p) * width).sum())


def work(case):
    names, _ = _ops(case)
    row = SIZE.get(case.get("dtype"), 0)
    if case["path"] == "scan":
        return {"bytes": case["rows"] * row + agg.SCALAR_BYTES, "flops": 0}
    if case["path"] == "packed":
        # i32 and i64 frames of values with about 17 and 21 bits of range, u32 with 16
        return {"bytes": case["rows"] * {"i32": 17, "u32": 16, "i64": 20}[case["dtype"]] / 8 + agg.SCALAR_BYTES, "flops": 0}
    if case["path"] == "batch":
        b = 0.0
        for j in range(BATCH_QUERIES):
            n = int(round(case["low"] * (case["rows"] / case["low"]) ** (j / (BATCH_QUERIES - 1)))) | 1
            count = max(1, min(n, int(round(case["keys"] ** (((5 * j) % BATCH_QUERIES) / (BATCH_QUERIES - 1))))))
            b += n * (4 + [4, 8, 4, 8][j % 4]) + _groups(n, count, [0.0, 1.0, 0.7][j % 3]) * (4 + 8 * len(names))
        return {"bytes": b, "flops": 0}
    return {"bytes": case["rows"] * (4 + row) + _groups(case["rows"], case["keys"], case["skew"]) * (4 + 8 * len(names)),
            "flops": 0}


# ---------------------------------------------------------------------------
# The float outputs in float64
# ---------------------------------------------------------------------------
def _wide(v):
    if v.dtype == torch.uint32:
        return v.view(torch.int32).to(torch.int64) & 0xFFFFFFFF
    return v.double() if v.is_floating_point() else v.to(torch.int64)


def _exact_scalar(col, names):
    v = _wide(col)
    fp = v.is_floating_point()
    s = v.sum()
    got = {COUNT: None, SUM: s if fp else None, AVG: s.double() / v.numel(), MIN: v.min() if fp else None,
           MAX: v.max() if fp else None}
    return {k: got[k] for k in names}


def _exact_groups(keys, vals, names):
    """Per distinct key (ascending): sums in float64 (or int64), extremes and averages."""
    uniq, inv = torch.unique(keys.view(torch.int32) ^ -0x80000000, return_inverse=True)  # unsigned order
    v = _wide(vals)
    fp, d = v.is_floating_point(), uniq.numel()
    out = {"keys": None}
    total = torch.zeros(d, dtype=v.dtype, device=v.device).index_add_(0, inv, v) if SUM in names or AVG in names else None
    for name in names:
        if name == SUM and fp:
            out[name] = total
        elif name == AVG:
            out[name] = total.double() / torch.bincount(inv, minlength=d).double()
        elif name in (MIN, MAX) and fp:
            start = math.inf if name == MIN else -math.inf
            out[name] = torch.full((d,), start, dtype=v.dtype, device=v.device).scatter_reduce_(
                0, inv, v, "amin" if name == MIN else "amax")
        else:
            out[name] = None
    return out


def exact(case, seed):
    names, _ = _ops(case)
    if case.get("dtype") not in (None, *FLOATS) and AVG not in names:
        return None  # whole numbers only
    if case["path"] == "scan":
        return _exact_scalar(_values(case["dtype"], case["rows"], seed), names)
    if case["path"] == "packed":
        return _exact_scalar(_packable(case, seed), names)
    if case["path"] == "batch":
        return [_exact_groups(k, v, names) for _, k, v in _queries(case, seed)]
    keys = _keys(case["rows"], case["keys"], case["skew"], seed)
    return _exact_groups(keys, _values(case["dtype"], case["rows"], seed), names)
