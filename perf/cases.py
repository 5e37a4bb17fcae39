"""What a user of this library has it do, as cases that can be timed.

The library runs query operators over columns in host memory, so most cases
hold their columns in page-locked host memory and time the whole call; the
allocation-free filter works on device columns.  Inputs follow the workloads
of this repository's benchmark and tests: the single-dimension query, the star
join templates over dimensions of 2,556 / 200,000 / 2,000,000 / 30,000 rows,
sorts of (uint64 key, uint32 row id) pairs that are uniform, Zipf(1.1) or made
of 64 presorted runs, and joins of unique 64-bit keys with uniform or Zipf(1.0)
probe keys at match rates 0.5 and 1.

listed() gives the cases, draw(rng) more of the same ranges, prepare(case, seed)
what a program has before the call, run(state) one call, work(case) the bytes
that it cannot do without and exact(case, seed) its outputs from plain torch.
"""
import math

import numpy as np
import torch

import paper_2502_09541_gb300 as vx

MIB = 1 << 20
DIM_ROWS = {"date": 2556, "supp": 200_000, "part": 2_000_000, "cust": 30_000}
ATTR_CARD = {
    "date": {"year": 7, "month": 12},
    "supp": {"region": 5, "nation": 25, "city": 250},
    "part": {"mfgr": 5, "category": 25, "brand": 250},
    "cust": {"region": 5, "nation": 25, "city": 250},
}
FACT_RANGE = {"date_fk": (0, 2555), "fk_supp": (0, 199_999), "fk_part": (0, 1_999_999), "fk_cust": (0, 29_999),
              "quantity": (1, 50), "discount": (0, 10), "price": (90_000, 10_000_000), "cost": (1_000, 100_000)}
I32MIN = -2**31


def _templates():
    """One-, three- and four-probe star queries at about 2, 0.1, 1 and 10 % selectivity."""
    t = {"T1": {"dims": [{"dim": "date", "fk": "date_fk", "preds": [("year", 1, 1)]}],
                "fact_preds": [("discount", 1, 3), ("quantity", I32MIN, 24)],
                "group": [], "agg": ("mul", "price", "discount")}}
    for sel, cat, reg, qty in (("10", 4, 2, 42), ("1", 1, 1, 16), ("0.1", 0, 0, 6)):
        t["T2_" + sel] = {"dims": [{"dim": "part", "fk": "fk_part", "preds": [("category", 0, cat)]},
                                   {"dim": "supp", "fk": "fk_supp", "preds": [("region", 0, reg)]},
                                   {"dim": "date", "fk": "date_fk", "preds": []}],
                          "fact_preds": [("quantity", I32MIN, qty)],
                          "group": [("date", "year"), ("part", "category")], "agg": ("sub", "price", "cost")}
    for sel, nat, year, disc in (("10", 11, 0, (0, 2)), ("1", 3, 4, (2, 3)), ("0.1", 0, 6, (2, 3))):
        t["T3_" + sel] = {"dims": [{"dim": "cust", "fk": "fk_cust", "preds": [("nation", 0, nat)]},
                                   {"dim": "supp", "fk": "fk_supp", "preds": []},
                                   {"dim": "date", "fk": "date_fk", "preds": [("year", year, 6)]},
                                   {"dim": "part", "fk": "fk_part", "preds": [("mfgr", 0, 3)]}],
                          "fact_preds": [("discount", disc[0], disc[1])],
                          "group": [("date", "year"), ("cust", "nation"), ("supp", "region")],
                          "agg": ("sub", "price", "cost")}
    return t


TEMPLATES = _templates()
SERVED = ("T1", "T2_10", "T2_1", "T2_0.1", "T3_10", "T3_1", "T3_0.1")


def listed():
    return [
        # a filter inside another program's latency path: one small batch of device rows, two predicates
        {"name": "filter_device_small", "kind": "filter", "rows": 10_007, "preds": 2, "sel": 0.13},
        # the same over the most rows a call takes (2^26), ragged, three predicates on three columns
        {"name": "filter_device_large", "kind": "filter", "rows": (1 << 26) - 1_003, "preds": 3, "sel": 0.02},
        # the single-dimension query as configured: 6,000,000 rows, 64 MiB budget, 8 MiB chunks
        {"name": "query_single_dim", "kind": "star", "rows": 6_000_000, "template": "T1", "batched": False,
         "budget_mib": 64, "chunk_mib": 8},
        # an ordinary star query, three probes at 1 % (late materialization), default executor settings
        {"name": "star_plain", "kind": "star", "rows": 60_000_001, "template": "T2_1", "batched": False,
         "budget_mib": 1024, "chunk_mib": 64},
        # the batched form of the benchmark on the largest fact table here: captured graph, copy-kernel
        # staging, per-chunk decisions, four probes at 10 %
        {"name": "star_batched", "kind": "star", "rows": (1 << 27) - 5, "template": "T3_10", "batched": True,
         "budget_mib": 4096, "chunk_mib": 256},
        # a burst of concurrent queries of uneven sizes at the serving engine
        {"name": "serve_burst", "kind": "serve", "rows": 30_000_000, "queries": 24, "budget_mib": 1024},
        # an in-memory sort of pairs from ordinary host arrays, odd size
        {"name": "sort_pairs", "kind": "pairs", "rows": 3_000_017, "dist": "uniform"},
        # out-of-core sort of full 64-bit keys, the default plan and splitters
        {"name": "sort_uniform", "kind": "sort", "rows": (1 << 26) - 1_001, "dist": "uniform", "plan": "partition",
         "partitioner": "sample", "budget_mib": 1024},
        # the learned form on skewed keys: the MLP partitioner, trained on each call's sample
        {"name": "sort_zipf_learned", "kind": "sort", "rows": 50_000_003, "dist": "zipf", "plan": "partition",
         "partitioner": "mlp", "budget_mib": 1024},
        # the merge plan on what it is for: an input already made of sorted runs
        {"name": "sort_runs_merge", "kind": "sort", "rows": 60_000_001, "dist": "runs", "plan": "merge",
         "partitioner": "sample", "budget_mib": 1024},
        # a join whose build table fits the budget, half of the probe keys without a match
        {"name": "join_direct", "kind": "join", "build": 8_000_000, "probe": (1 << 26) - 9, "match": 0.5, "zipf": False,
         "algorithm": "direct", "budget_mib": 2048},
        # the radix-partitioned join, skewed probe keys
        {"name": "join_radix", "kind": "join", "build": 3_000_000, "probe": 30_000_001, "match": 1.0, "zipf": True,
         "algorithm": "radix", "budget_mib": 2048},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["filter", "filter", "star", "star", "serve", "pairs", "sort", "sort", "join"])
    if kind == "filter":
        return {"kind": kind, "rows": _log(rng, 300, 1 << 26), "preds": rng.randint(1, 4),
                "sel": round(10 ** rng.uniform(-3, -0.05), 4)}
    if kind == "star":
        rows = _log(rng, 1_000_000, (1 << 27) - 5)
        batched = rng.random() < 0.5
        budget = rng.choice([512, 1024, 4096])
        return {"kind": kind, "rows": rows, "template": rng.choice(SERVED), "batched": batched, "budget_mib": budget,
                "chunk_mib": rng.choice([16, 64] if budget < 4096 else [64, 256])}
    if kind == "serve":
        return {"kind": kind, "rows": _log(rng, 5_000_000, 30_000_000), "queries": rng.randint(4, 24), "budget_mib": 1024}
    if kind == "pairs":
        return {"kind": kind, "rows": _log(rng, 1_000, 8_000_000), "dist": rng.choice(["uniform", "zipf", "runs"])}
    if kind == "sort":
        return {"kind": kind, "rows": _log(rng, 4_000_000, (1 << 26) - 1_001), "dist": rng.choice(["uniform", "zipf", "runs"]),
                "plan": rng.choice(["partition", "partition", "merge"]), "partitioner": rng.choice(["sample", "pl", "mlp"]),
                "budget_mib": rng.choice([256, 1024, 3072])}
    direct = rng.random() < 0.6
    top = 8_000_000 if direct else 3_000_000
    return {"kind": "join", "build": _log(rng, 500_000, top), "probe": _log(rng, 4_000_000, 8 * top),
            "match": rng.choice([0.5, 1.0]), "zipf": rng.random() < 0.5, "algorithm": "direct" if direct else "radix",
            "budget_mib": 2048}


# ---------------------------------------------------------------- inputs, made on the GPU
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1_000_003 + salt)
    return g


def _ints(n, lo, hi, g):
    return torch.randint(lo, hi + 1, (n,), dtype=torch.int32, device="cuda", generator=g)


def _host(t, pinned=True):
    """The tensor's values in host memory, page-locked as a streaming program keeps its columns."""
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=pinned)
    h.copy_(t)
    return h


def _shr(x, k):
    return (x >> k) & ((1 << (64 - k)) - 1)


def _mix64(x):
    """The SplitMix64 finalizer on int64 tensors (wrapping)."""
    x = (x ^ _shr(x, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    x = (x ^ _shr(x, 27)) * (0x94D049BB133111EB - (1 << 64))
    return x ^ _shr(x, 31)


def _zipf(n, ranks, s, g):
    """Ranks in [0, ranks) with density falling as (rank + 1)^-s."""
    u = torch.rand(n, dtype=torch.float64, device="cuda", generator=g)
    if s == 1.0:
        x = torch.exp(u * math.log(ranks + 1.0))
    else:
        x = (1.0 + u * ((ranks + 1.0) ** (1.0 - s) - 1.0)) ** (1.0 / (1.0 - s))
    return (x.to(torch.int64) - 1).clamp_(0, ranks - 1)


def _pairs(case, seed):
    """(keys as int64 bits, row ids as int32 bits) on the GPU."""
    n, g = case["rows"], _gen(seed, 1)
    if case["dist"] == "zipf":
        k = _mix64(_zipf(n, 1 << 30, 1.1, g))
    else:
        k = torch.randint(-2**63, 2**63 - 1, (n,), dtype=torch.int64, device="cuda", generator=g)
        if case["dist"] == "runs":
            cut = [n * r // 64 for r in range(65)]
            for a, b in zip(cut, cut[1:]):
                k[a:b] = _unsigned_sort(k[a:b])[0]
    return k, torch.arange(n, dtype=torch.int32, device="cuda")


def _unsigned_sort(k):
    s, at = torch.sort(k ^ -2**63, stable=True)
    return s ^ -2**63, at


def _filter_preds(case):
    """Predicates (column, op, lo, hi) on columns of 0 .. 999,999 that together pass about sel of the rows."""
    each = case["sel"] ** (1.0 / case["preds"])
    w = max(1, min(999_999, int(each * 1_000_000)))
    kinds = [(vx.VX_LT, w, 0), (vx.VX_BETWEEN, 1_000, 1_000 + w - 1), (vx.VX_GE, 1_000_000 - w, 0), (vx.VX_LE, w - 1, 0)]
    return [(q, *kinds[q]) for q in range(case["preds"])]


def _filter_cols(case, seed):
    g = _gen(seed, 2)
    return [_ints(case["rows"], 0, 999_999, g) for _ in range(case["preds"])]


def _star_columns(case):
    names = ("date_fk", "fk_supp", "fk_part", "fk_cust", "quantity", "discount", "price", "cost")
    if case["kind"] == "serve":
        return names
    t = TEMPLATES[case["template"]]
    used = {d["fk"] for d in t["dims"]} | {p[0] for p in t["fact_preds"]} | {c for c in t["agg"][1:] if c}
    return tuple(c for c in names if c in used)


def _star_tables(case, seed):
    """(fact columns, dimensions) on the GPU."""
    g = _gen(seed, 3)
    fact = {c: _ints(case["rows"], *FACT_RANGE[c], g) for c in _star_columns(case)}
    dims = {}
    for name, rows in DIM_ROWS.items():
        d = {"key": torch.randperm(rows, device="cuda", generator=g).to(torch.int32)}
        a = list(ATTR_CARD[name])
        if name == "date":  # 2,556 days from 1992 on, kept as year and month codes
            d["year"] = torch.clamp(d["key"] // 365, max=6)
            d["month"] = torch.clamp(d["key"] % 365 // 31, max=11)
        else:  # region -> nation -> city style codes
            d[a[0]] = _ints(rows, 0, 4, g)
            d[a[1]] = d[a[0]] * 5 + _ints(rows, 0, 4, g)
            d[a[2]] = d[a[1]] * 10 + _ints(rows, 0, 9, g)
        dims[name] = {k: v.to(torch.int32) for k, v in d.items()}
    return fact, dims


def _join_tables(case, seed):
    """(build keys, build payload, probe keys, build row of each probe or -1) on the GPU."""
    nb, n, g = case["build"], case["probe"], _gen(seed, 4)
    i = torch.arange(nb, dtype=torch.int64, device="cuda") + seed * (1 << 32)
    keys, pay = _mix64(i), _mix64(i ^ 0x5DEECE66D)
    if case["zipf"]:
        at = (_zipf(n, nb, 1.0, g) * 2_654_435_761 + 12_345) % nb
    else:
        at = torch.randint(0, nb, (n,), dtype=torch.int64, device="cuda", generator=g)
    miss = torch.rand(n, device="cuda", generator=g) >= case["match"]
    probe = torch.where(miss, _mix64(at + seed * (1 << 32) + (1 << 31)), keys[at])
    return keys, pay, probe, torch.where(miss, -1, at)


def _served(case, seed):
    """(template, first row, end row) of each query: sizes log-uniform up to the whole table."""
    r = np.random.default_rng(seed)
    got = []
    for _ in range(case["queries"]):
        size = int(np.exp(r.uniform(np.log(100_000), np.log(case["rows"]))))
        at = int(r.integers(0, case["rows"] - size + 1))
        got.append((SERVED[int(r.integers(0, len(SERVED)))], at, at + size))
    return got


# ---------------------------------------------------------------- what a program holds
class Session:
    """An open context and the host arrays whose columns it has registered."""

    def __init__(self, budget_mib, **config):
        self.keep = []
        self.ctx = vx.vx_open(budget_mib * MIB)
        if config:
            cfg = vx.vx_get_config(self.ctx)
            for k, v in config.items():
                setattr(cfg, k, v)
            vx.vx_set_config(self.ctx, cfg)

    def column(self, name, t, dtype):
        h = _host(t)
        self.keep.append(h)
        return vx.vx_register_host_column(self.ctx, name, h.numpy().view(dtype))

    def __del__(self):
        if getattr(self, "ctx", None):
            vx.vx_close(self.ctx)
            self.ctx = None


def _star_session(case, seed, **config):
    s = Session(case["budget_mib"], **config)
    fact, dims = _star_tables(case, seed)
    fid = {c: s.column(c, t, np.int32) for c, t in fact.items()}
    did = {d: {a: s.column(d + "." + a, t, np.int32) for a, t in v.items()} for d, v in dims.items()}
    return s, fid, did


def _empty(n, dtype):
    return torch.empty(n, dtype=dtype, pin_memory=True)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "filter":
        cols = _filter_cols(case, seed)
        return {"kind": kind, "cols": cols, "preds": _filter_preds(case), "n": case["rows"],
                "out": torch.full((case["rows"],), -1, dtype=torch.int64, device="cuda")}
    if kind == "star":
        late = vx.VX_LATE_PER_CHUNK if case["batched"] else vx.VX_LATE_AUTO
        s, fid, did = _star_session(case, seed, chunk_bytes=case["chunk_mib"] * MIB)
        tmpl = TEMPLATES[case["template"]]
        if case["batched"]:
            # the regressor is trained once on a logged plain run, then the pipeline is captured
            cfg = vx.vx_get_config(s.ctx)
            cfg.log_chunk_stats, cfg.chunk_bytes = 1, 8 * MIB
            vx.vx_set_config(s.ctx, cfg)
            vx.vx_run_plan(s.ctx, vx.make_plan(tmpl, fid, did, ATTR_CARD, vx.VX_LATE_AUTO, 0, min(case["rows"], 8_000_000)))
            vx.vx_regressor_train(s.ctx)
            cfg.log_chunk_stats, cfg.chunk_bytes = 0, case["chunk_mib"] * MIB
            cfg.use_graphs, cfg.h2d_copy_blocks = 1, 32
            vx.vx_set_config(s.ctx, cfg)
        return {"kind": kind, "session": s, "cells": _cells(tmpl), "plan": vx.make_plan(tmpl, fid, did, ATTR_CARD, late)}
    if kind == "serve":
        s, fid, did = _star_session(case, seed)
        plans = [vx.make_plan(TEMPLATES[t], fid, did, ATTR_CARD, vx.VX_LATE_AUTO, a, b) for t, a, b in _served(case, seed)]
        vx.vx_serve_start(s.ctx)
        return {"kind": kind, "session": s, "plans": plans}
    if kind == "pairs":
        k, r = _pairs(case, seed)
        kb = (8 * case["rows"] + 4 * case["rows"]) * 2
        return {"kind": kind, "session": Session(max(64, kb * 2 // MIB)), "keys": k.cpu().numpy().view(np.uint64),
                "vals": r.cpu().numpy().view(np.uint32)}
    if kind == "sort":
        n = case["rows"]
        s = Session(case["budget_mib"])
        k, r = _pairs(case, seed)
        o = vx.vx_sort_opts()
        o.plan = vx.VX_SORT_MERGE if case["plan"] == "merge" else vx.VX_SORT_PARTITION
        o.partitioner = {"sample": vx.VX_PART_SAMPLE, "pl": vx.VX_PART_LEARNED_PL, "mlp": vx.VX_PART_LEARNED_MLP}[case["partitioner"]]
        scratch = _empty(12 * (n + n // 8 + 65_536), torch.uint8)  # the intermediate, kept between calls
        o.host_scratch, o.host_scratch_bytes = scratch.data_ptr(), scratch.numel()
        return {"kind": kind, "session": s, "scratch": scratch, "opts": o, "key": s.column("key", k, np.uint64),
                "row": s.column("row", r, np.uint32), "out_k": _empty(n, torch.int64), "out_r": _empty(n, torch.int32)}
    s = Session(case["budget_mib"])
    keys, pay, probe, _ = _join_tables(case, seed)
    o = vx.vx_join_opts()
    o.algorithm = vx.VX_JOIN_RADIX if case["algorithm"] == "radix" else vx.VX_JOIN_DIRECT
    return {"kind": kind, "session": s, "opts": o, "bk": s.column("key", keys, np.int64),
            "bp": s.column("payload", pay, np.int64), "pk": s.column("probe", probe, np.int64)}


def _cells(tmpl):
    return math.prod(ATTR_CARD[d][a] for d, a in tmpl["group"])


def _table(cells, *results):
    """The queries' groups as (sum, count) tables over all group ids, as a report prints them."""
    sums, counts = np.zeros((len(results), cells), np.int64), np.zeros((len(results), cells), np.int64)
    for i, (gid, s, c) in enumerate(results):
        at = gid.view(np.int64)
        sums[i, at], counts[i, at] = s, c.view(np.int64)
    return sums, counts


def run(state):
    kind = state["kind"]
    if kind == "filter":
        # the call returns once the stream's work is done
        _, n = vx.vx_filter_device_static([c.data_ptr() for c in state["cols"]], state["preds"], state["n"], 0,
                                          state["out"].data_ptr(), state["n"], torch.cuda.current_stream().cuda_stream)
        return state["out"], n
    ctx = state["session"].ctx
    if kind == "star":
        _, gid, s, c, _ = vx.vx_run_plan(ctx, state["plan"], 1 << 13)
        return _table(state["cells"], (gid, s, c))
    if kind == "serve":
        tickets = [vx.vx_submit(ctx, p) for p in state["plans"]]
        got = [vx.vx_wait(ctx, t) for t in tickets]
        return _table(max(map(_cells, TEMPLATES.values())), *(g[1:4] for g in got))
    if kind == "pairs":
        k, v = vx.vx_radix_sort_pairs(ctx, state["keys"], state["vals"])
        return k.view(np.int64), v.view(np.int32)
    if kind == "sort":
        vx.vx_sort(ctx, state["key"], state["row"], state["out_k"].numpy(), state["out_r"].numpy(), state["opts"])
        return state["out_k"], state["out_r"]
    r = vx.vx_join(ctx, state["bk"], state["bp"], state["pk"], state["opts"])
    return np.array([r["count"], r["payload_sum"], r["pair_fp"]], np.uint64).view(np.int64)


def work(case):
    """Bytes: every input column once (over the host link, but for the device filter) and every output once."""
    kind = case["kind"]
    if kind == "filter":
        return {"bytes": case["rows"] * (4 * case["preds"] + 8 * case["sel"]), "flops": 0}
    if kind == "star":
        return {"bytes": 4 * case["rows"] * len(_star_columns(case)), "flops": 0}
    if kind == "serve":  # the table once, shared by all queries
        return {"bytes": 4 * case["rows"] * len(_star_columns(case)), "flops": 0}
    if kind in ("pairs", "sort"):
        return {"bytes": 24 * case["rows"], "flops": 0}
    return {"bytes": 16 * case["build"] + 8 * case["probe"], "flops": 0}


# ---------------------------------------------------------------- the same from plain torch
def _star_exact(tmpl, fact, dims, a, b, cells):
    """(sums, counts) of all groups over fact rows [a, b), `cells` of each."""
    col = {c: t[a:b] for c, t in fact.items()}
    keep = torch.ones(b - a, dtype=torch.bool, device="cuda")
    for c, lo, hi in tmpl["fact_preds"]:
        keep &= (col[c] >= lo) & (col[c] <= hi)
    at = torch.nonzero(keep).squeeze(1)
    rows = {}
    for d in tmpl["dims"]:
        dim = dims[d["dim"]]
        where = torch.empty(len(dim["key"]), dtype=torch.int64, device="cuda")
        where[dim["key"].long()] = torch.arange(len(dim["key"]), device="cuda")
        ok = torch.ones(len(dim["key"]), dtype=torch.bool, device="cuda")
        for attr, lo, hi in d["preds"]:
            ok &= (dim[attr] >= lo) & (dim[attr] <= hi)
        hit = where[col[d["fk"]][at].long()]
        good = ok[hit]
        at, rows = at[good], {k: v[good] for k, v in rows.items()}
        rows[d["dim"]] = hit[good]
    gid = torch.zeros(len(at), dtype=torch.int64, device="cuda")
    for d, attr in tmpl["group"]:
        gid = gid * ATTR_CARD[d][attr] + dims[d][attr][rows[d]]
    op, ca, cb = tmpl["agg"]
    x, y = col[ca][at].long(), col[cb][at].long()
    v = x * y if op == "mul" else x - y
    s = torch.zeros(cells, dtype=torch.int64, device="cuda").index_add_(0, gid, v)
    c = torch.zeros(cells, dtype=torch.int64, device="cuda").index_add_(0, gid, torch.ones_like(gid))
    return s, c


def exact(case, seed):
    kind = case["kind"]
    if kind == "filter":
        keep = torch.ones(case["rows"], dtype=torch.bool, device="cuda")
        for (_, op, lo, hi), c in zip(_filter_preds(case), _filter_cols(case, seed)):
            keep &= {vx.VX_LT: c < lo, vx.VX_BETWEEN: (c >= lo) & (c <= hi), vx.VX_GE: c >= lo, vx.VX_LE: c <= lo}[op]
        rows = torch.nonzero(keep).squeeze(1)
        return torch.nn.functional.pad(rows, (0, case["rows"] - len(rows)), value=-1), len(rows)
    if kind == "star":
        tmpl = TEMPLATES[case["template"]]
        s, c = _star_exact(tmpl, *_star_tables(case, seed), 0, case["rows"], _cells(tmpl))
        return s[None], c[None]
    if kind == "serve":
        fact, dims = _star_tables(case, seed)
        cells = max(map(_cells, TEMPLATES.values()))
        got = [_star_exact(TEMPLATES[t], fact, dims, a, b, cells) for t, a, b in _served(case, seed)]
        return tuple(torch.stack([g[k] for g in got]) for k in range(2))
    if kind in ("pairs", "sort"):
        k, r = _pairs(case, seed)
        k, at = _unsigned_sort(k)
        return k, r[at]
    _, pay, _, at = _join_tables(case, seed)
    row = torch.nonzero(at >= 0).squeeze(1)
    p = pay[at[row]]
    fp = _mix64(row ^ ((p << 17) | _shr(p, 47)))
    return torch.stack([torch.tensor(len(row), device="cuda"), p.sum(), fp.sum()])
