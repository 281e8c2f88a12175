"""The work this library is timed on: its operators and queries as a program calls them.

Sizes, value ranges and distributions are those of the repository's own workloads
(``bench.py``, ``datagen``, ``tests``): selection and projection of columns up to 2^29
rows, joins of 2^10 to 2^27 build rows with up to 2^28 probe rows, sorts up to 2^28
pairs, the fused date-join query from 2^22 rows, and select-join-group-by queries over
the star schema (600M fact rows, dimensions of 2556 / 200K / 3M / 1.4M rows) alone and
as batches of 32 that share one scan.  A state holds the columns in device memory and
whatever a program keeps between calls (a loaded star schema, a dimension table, the
output buffer of a selection, whose rows past the count stay 0); a pass is the whole
call, with the outputs and scratch that the library's wrappers allocate for any user.  Integer results are exact; the unstable sort gets distinct keys and the
order-free selection equal values, so that their results are unique.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2003_01178_gb300 as crys
from paper_2003_01178_gb300.starschema import ResidentStarSchema, Schema

I32_MIN, I32_MAX = -(1 << 31), (1 << 31) - 1
DEVICE = "cuda"

DIMS = {
    "date": {"rows": 2556, "fk": "fk_date", "attrs": {"year": 7, "month": 12}},
    "supp": {"rows": 200_000, "fk": "fk_supp", "attrs": {"region": 5, "nation": 25, "city": 250}},
    "cust": {"rows": 3_000_000, "fk": "fk_cust", "attrs": {"region": 5, "nation": 25, "city": 250}},
    "part": {"rows": 1_400_000, "fk": "fk_part", "attrs": {"mfgr": 5, "category": 25, "brand": 1000}},
}
MEASURES = {"qty": (1, 50), "disc": (0, 10), "price": (1, 100_000), "cost": (1, 60_000)}
FACT_COLS = [s["fk"] for s in DIMS.values()] + list(MEASURES)
GROUP_LIMIT = 10_000


def listed() -> list:
    return [
        # a small filtered column in row order: launches count
        {"name": "select_small", "op": "select", "n": 100_003, "sigma": 0.5, "ordered": True},
        # a full column filtered to half, in row order (late materialisation, exports)
        {"name": "select_large", "op": "select", "n": 1 << 29, "sigma": 0.5, "ordered": True},
        # a computed float column: the sigmoid of a linear combination
        {"name": "project_large", "op": "project", "n": (1 << 28) + 3, "sigmoid": True},
        # a date-sized dimension joined to a small fact table, table built in the query
        {"name": "join_small", "op": "join", "nb": 2556, "np": 1_000_003, "match": 1.0},
        # a dimension whose table lives in L2, a fact table far beyond it
        {"name": "join_large", "op": "join", "nb": 1 << 22, "np": 1 << 28, "match": 1.0},
        # both sides far beyond the caches: the radix-partitioned join
        {"name": "join_partitioned", "op": "join_part", "nb": 1 << 27, "np": 1 << 28, "match": 1.0},
        # a small result set put in order (ORDER BY of a query's output)
        {"name": "sort_small", "op": "sort", "n": 100_003, "keys": "bits"},
        # a full column of pairs, stable
        {"name": "sort_large", "op": "sort", "n": 1 << 28, "keys": "bits"},
        # the same size by the unstable most-significant-digit sort
        {"name": "sort_msb_large", "op": "sort_msb", "n": 1 << 28, "keys": "bits"},
        # one selective date-join query over a small fact table
        {"name": "query_small", "op": "query", "n": 1 << 22, "a_max": 24},
        # one grouped three-join query over a fact table of SSB's scale factor 10
        {"name": "query_star", "op": "star", "n": 60_000_003, "queries": 1, "joins": 3, "qseed": 11},
        # a served batch: 32 queries of the stream in one shared scan of the whole table
        {"name": "batch_star", "op": "star", "n": 600_000_000, "queries": 32, "joins": 0, "qseed": 1},
    ]


def _log_uniform(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random) -> dict:
    op = rng.choice(["select", "project", "join", "join", "join_part", "sort", "sort", "sort_msb", "query", "star", "star"])
    if op == "select":
        return {"op": op, "n": _log_uniform(rng, 1_000, 1 << 29), "sigma": round(rng.random(), 3),
                "ordered": rng.random() < 0.6}
    if op == "project":
        return {"op": op, "n": _log_uniform(rng, 1_000, 1 << 28), "sigmoid": rng.random() < 0.5}
    if op == "join":
        return {"op": op, "nb": _log_uniform(rng, 1 << 8, 1 << 26), "np": _log_uniform(rng, 10_000, 1 << 28),
                "match": rng.choice([1.0, 0.5, 0.1])}
    if op == "join_part":
        nb = _log_uniform(rng, 1 << 12, 1 << 27)
        return {"op": op, "nb": nb, "np": _log_uniform(rng, 1 << 16, 1 << 28), "match": rng.choice([1.0, 0.5])}
    if op == "sort":
        # raw patterns, foreign keys into a dimension a fifth as long, or a low-cardinality code
        return {"op": op, "n": _log_uniform(rng, 100, 1 << 28), "keys": rng.choice(["bits", "bits", "dense", "few"])}
    if op == "sort_msb":
        keys = rng.choice(["bits", "bits", "dense"])
        return {"op": op, "n": _log_uniform(rng, 100, 1 << 28 if keys == "bits" else 1 << 25), "keys": keys}
    if op == "query":
        return {"op": op, "n": _log_uniform(rng, 1 << 18, 1 << 28), "a_max": rng.choice([1, 24, 50])}
    queries = rng.choice([1, 1, 4, 8, 16, 32])
    return {"op": op, "n": _log_uniform(rng, 1_000_000, 300_000_000), "queries": queries,
            "joins": rng.randint(1, 4) if queries == 1 else 0, "qseed": rng.randint(0, 1 << 20)}


# ---------------------------------------------------------------------------- inputs

def _gen(seed: int, stream: int) -> torch.Generator:
    g = torch.Generator(device=DEVICE)
    g.manual_seed((seed * 1_000_003 + stream) & ((1 << 62) - 1))
    return g


def _uniform(seed: int, stream: int, n: int, lo: int, hi: int) -> torch.Tensor:
    """n int32 values uniform in [lo, hi]."""
    return torch.randint(lo, hi + 1, (n,), dtype=torch.int32, device=DEVICE, generator=_gen(seed, stream))


def _perm(seed: int, stream: int, n: int) -> torch.Tensor:
    return torch.randperm(n, device=DEVICE, generator=_gen(seed, stream)).to(torch.int32)


def _bits(seed: int, stream: int, n: int) -> torch.Tensor:
    """n int32 values over the whole range."""
    return torch.randint(I32_MIN, I32_MAX + 1, (n,), dtype=torch.int64, device=DEVICE,
                         generator=_gen(seed, stream)).to(torch.int32)


def _distinct_bits(seed: int, n: int) -> torch.Tensor:
    """n distinct int32 values spread over the whole range: a 32-bit bijection (xor-shifts
    and odd multiplications) of the counters seed .. seed + n - 1."""
    x = (torch.arange(n, dtype=torch.int64, device=DEVICE) + seed * 0x9E3779B1) & 0xFFFFFFFF
    for mult in (0x7FEB352D, 0x846CA68B):
        x ^= x >> 16
        x *= mult
        x &= 0xFFFFFFFF
        x ^= x >> 15
    return x.to(torch.int32)


def _sort_keys(case: dict, seed: int) -> torch.Tensor:
    n = case["n"]
    if case["op"] == "sort_msb":
        return _distinct_bits(seed, n) if case["keys"] == "bits" else _perm(seed, 1, n)
    if case["keys"] == "bits":
        return _bits(seed, 1, n)
    return _uniform(seed, 1, n, 0, max(1, n // 5) if case["keys"] == "dense" else 49)


def _threshold(sigma: float) -> int:
    return min(int(round(sigma * (1 << 31))) - 1, I32_MAX)


def _select_input(case: dict, seed: int):
    """(column, lo, hi): a range of uniform values in row order, or one value of a column
    of 50 (a quantity) without an order."""
    if case["ordered"]:
        return _uniform(seed, 1, case["n"], 0, I32_MAX), I32_MIN, _threshold(case["sigma"])
    return _uniform(seed, 1, case["n"], 1, 50), 24, 24


def _join_input(case: dict, seed: int):
    nb, n_probe = case["nb"], case["np"]
    last = max(nb, int(nb / case["match"])) - 1
    return (_perm(seed, 1, nb), _uniform(seed, 2, nb, 1, 100), _uniform(seed, 3, n_probe, 0, last),
            _uniform(seed, 4, n_probe, 1, 100))


def _query_input(case: dict, seed: int):
    n = case["n"]
    fact = [_uniform(seed, 1, n, 0, 2555), _uniform(seed, 2, n, 1, 50), _uniform(seed, 3, n, 0, 10),
            _uniform(seed, 4, n, 1, 100_000)]
    key = _perm(seed, 5, 2556)
    year = (torch.arange(2556, device=DEVICE) % 7).to(torch.int32)
    return fact, key, year


def _star_input(case: dict, seed: int):
    n = case["n"]
    fact = {}
    for i, c in enumerate(FACT_COLS):
        lo, hi = MEASURES[c] if c in MEASURES else (0, next(s["rows"] for s in DIMS.values() if s["fk"] == c) - 1)
        fact[c] = _uniform(seed, 10 + i, n, lo, hi)
    dims = {}
    for d, (name, spec) in enumerate(DIMS.items()):
        dims[name] = {"key": _perm(seed, 50 + 10 * d, spec["rows"])}
        for a, (attr, card) in enumerate(spec["attrs"].items()):
            dims[name][attr] = _uniform(seed, 51 + 10 * d + a, spec["rows"], 0, card - 1)
    return fact, dims


def _queries(case: dict) -> list:
    """Seeded select-join-group-by queries: 1 to 4 joins, selectivity log-uniform in
    [1e-4, 0.5], at most 10^4 groups, a quantity range in a quarter of them."""
    out = []
    for q in range(case["queries"]):
        rng = random.Random(case["qseed"] * 64 + q)
        k = case["joins"] or rng.randint(1, 4)
        target = math.exp(rng.uniform(math.log(1e-4), math.log(0.5)))
        joins, groups = [], 1
        for d in rng.sample(list(DIMS), k):
            attrs = DIMS[d]["attrs"]
            name = rng.choice(list(attrs))
            width = max(1, min(attrs[name], int(round(target ** (1.0 / k) * attrs[name]))))
            lo = rng.randint(0, attrs[name] - width)
            group = rng.choice([None] + list(attrs))
            if group is not None and groups * attrs[group] > GROUP_LIMIT:
                group = None
            if group is not None:
                groups *= attrs[group]
            joins.append({"dim": d, "filters": [(name, lo, lo + width - 1)] if width < attrs[name] else [],
                          "group": group})
        preds = []
        if rng.random() < 0.25:
            lo = rng.randint(1, 25)
            preds = [("qty", lo, lo + 24)]
        agg = rng.choice([("mul", "price", "disc"), ("sum", "price", None), ("sub", "price", "cost")])
        out.append({"id": q, "fact_preds": preds, "joins": joins, "agg": agg})
    return out


# ---------------------------------------------------------------------------- the calls

def prepare(case: dict, seed: int) -> dict:
    op = case["op"]
    st = {"op": op, "case": case}
    if op == "select":
        st["x"], st["lo"], st["hi"] = _select_input(case, seed)
        # the caller's own output buffer, count and (for row order) scratch, kept between calls
        st["out"] = torch.zeros(case["n"], dtype=torch.int32, device=DEVICE)
        st["count"] = torch.zeros(1, dtype=torch.int64, device=DEVICE)
        st["temp"], st["temp_bytes"] = None, None
        if case["ordered"]:
            st["temp_bytes"] = crys.crys_select(None, case["n"], st["lo"], st["hi"], None, None, 1, None, -1)
            st["temp"] = crys.scratch(st["temp_bytes"], DEVICE)
    elif op == "project":
        st["x1"] = torch.rand(case["n"], device=DEVICE, generator=_gen(seed, 1))
        st["x2"] = torch.rand(case["n"], device=DEVICE, generator=_gen(seed, 2))
    elif op in ("join", "join_part"):
        st["bk"], st["bv"], st["fk"], st["pay"] = _join_input(case, seed)
    elif op in ("sort", "sort_msb"):
        st["keys"] = _sort_keys(case, seed)
        st["vals"] = torch.arange(case["n"], dtype=torch.int32, device=DEVICE)
    elif op == "query":
        fact, key, year = _query_input(case, seed)
        st["fact"] = fact
        st["table"] = crys.HashTable.build(key, year, filters=[(year, 3, 3)], capacity=2556, kind=crys.HASH_DIRECT)
    else:
        fact, dims = _star_input(case, seed)
        st["store"] = ResidentStarSchema(Schema.from_spec(FACT_COLS, DIMS), fact, dims)
        st["queries"] = _queries(case)
    return st


def run(st: dict):
    op, case = st["op"], st["case"]
    if op == "select":
        crys.crys_select(st["x"], case["n"], st["lo"], st["hi"], st["out"], st["count"], int(case["ordered"]),
                         st["temp"], st["temp_bytes"])
        return st["out"], st["count"]
    if op == "project":
        return crys.project(st["x1"], st["x2"], 2.0, 3.0, crys.PROJ_SIGMOID if case["sigmoid"] else crys.PROJ_LINEAR)
    if op == "join":
        return crys.probe_aggregate(st["fk"], st["pay"], crys.HashTable.build(st["bk"], st["bv"]))
    if op == "join_part":
        return crys.join_partitioned(st["bk"], st["bv"], st["fk"], st["pay"])
    if op == "sort":
        return crys.sort(st["keys"], st["vals"])
    if op == "sort_msb":
        return crys.sort_msb(st["keys"], st["vals"])
    if op == "query":
        return crys.run_plan(st["fact"], [(1, I32_MIN, case["a_max"]), (2, 1, 3)], [(0, st["table"], 0)], ("mul", 3, 2))
    store = st["store"]
    cqs = [store.compile(q) for q in st["queries"]]
    if len(cqs) == 1:
        store.run(cqs[0])
    else:
        store.run_shared(cqs)
    return [(c.sums, c.counts) for c in cqs]


# ---------------------------------------------------------------------------- what is needed, and what is right

def work(case: dict) -> dict:
    op = case["op"]
    if op == "select":
        n = case["n"]
        return {"bytes": 4 * n * (1 + (case["sigma"] if case["ordered"] else 0.02)), "flops": 0}
    if op == "project":
        return {"bytes": 12 * case["n"], "flops": (6 if case["sigmoid"] else 3) * case["n"]}
    if op in ("join", "join_part"):
        return {"bytes": 8 * (case["nb"] + case["np"]), "flops": 2 * case["np"]}
    if op in ("sort", "sort_msb"):
        return {"bytes": 16 * case["n"], "flops": 0}
    if op == "query":
        return {"bytes": 16 * case["n"], "flops": 2 * case["n"]}
    queries = _queries(case)
    cols, dims, groups = set(), set(), 0
    for q in queries:
        cols |= {c for c, _, _ in q["fact_preds"]} | {DIMS[j["dim"]]["fk"] for j in q["joins"]}
        cols |= {c for c in q["agg"][1:] if c is not None}
        dims |= {j["dim"] for j in q["joins"]}
        groups += math.prod(DIMS[j["dim"]]["attrs"][j["group"]] for j in q["joins"] if j["group"])
    return {"bytes": 4 * case["n"] * len(cols) + sum(8 * DIMS[d]["rows"] for d in dims) + 16 * groups,
            "flops": 2 * case["n"]}


def _exact_join(case: dict, seed: int):
    bk, bv, fk, pay = _join_input(case, seed)
    value = torch.zeros(case["nb"], dtype=torch.int64, device=DEVICE)
    value[bk.long()] = bv.long()
    total = torch.zeros(1, dtype=torch.int64, device=DEVICE)
    matches = torch.zeros(1, dtype=torch.int64, device=DEVICE)
    for b in range(0, case["np"], 1 << 26):
        k, p = fk[b:b + (1 << 26)].long(), pay[b:b + (1 << 26)].long()
        hit = k < case["nb"]
        total += (p[hit] * value[k[hit]]).sum()
        matches += hit.sum()
    return total, matches


def _exact_query(case: dict, seed: int):
    (fk, a, b, c), key, year = _query_input(case, seed)
    by_key = torch.zeros(2556, dtype=torch.int32, device=DEVICE)
    by_key[key.long()] = year
    hit = (a <= case["a_max"]) & (b >= 1) & (b <= 3) & (by_key[fk.long()] == 3)
    return (c[hit].long() * b[hit].long()).sum().reshape(1), hit.sum().reshape(1)


def _exact_star(case: dict, seed: int):
    fact, dims = _star_input(case, seed)
    by_key = {}
    for d, cols in dims.items():
        for attr in DIMS[d]["attrs"]:
            v = torch.empty_like(cols[attr])
            v[cols["key"].long()] = cols[attr]
            by_key[d, attr] = v
    out = []
    for q in _queries(case):
        groups = math.prod(DIMS[j["dim"]]["attrs"][j["group"]] for j in q["joins"] if j["group"])
        out.append((torch.zeros(groups, dtype=torch.int64, device=DEVICE),
                    torch.zeros(groups, dtype=torch.int64, device=DEVICE)))
    step = 1 << 25
    for b in range(0, case["n"], step):
        part = {c: v[b:b + step] for c, v in fact.items()}
        for q, (sums, counts) in zip(_queries(case), out):
            rows = None
            for c, lo, hi in q["fact_preds"]:
                rows = ((part[c] >= lo) & (part[c] <= hi)).nonzero().flatten()
            for j in q["joins"]:
                for attr, lo, hi in j["filters"]:
                    fk = part[DIMS[j["dim"]]["fk"]]
                    v = by_key[j["dim"], attr][(fk if rows is None else fk[rows]).long()]
                    keep = ((v >= lo) & (v <= hi)).nonzero().flatten()
                    rows = keep if rows is None else rows[keep]
            rows = slice(None) if rows is None else rows
            gid = torch.zeros(1, dtype=torch.int64, device=DEVICE)
            for j in q["joins"]:
                if j["group"]:
                    code = by_key[j["dim"], j["group"]][part[DIMS[j["dim"]]["fk"]][rows].long()]
                    gid = gid * DIMS[j["dim"]]["attrs"][j["group"]] + code
            op, x, y = q["agg"]
            val = part[x][rows].long()
            if op == "mul":
                val = val * part[y][rows].long()
            elif op == "sub":
                val = val - part[y][rows].long()
            gid = gid.expand(val.numel())
            sums.index_add_(0, gid, val)
            counts.index_add_(0, gid, torch.ones_like(val))
    return out


def exact(case: dict, seed: int):
    op = case["op"]
    if op == "select":
        x, lo, hi = _select_input(case, seed)
        kept = x[(x >= lo) & (x <= hi)]
        out = torch.zeros_like(x)
        out[:kept.numel()] = kept
        return out, torch.tensor([kept.numel()], dtype=torch.int64, device=DEVICE)
    if op == "project":
        st = prepare(case, seed)
        lin = 2.0 * st["x1"].double() + 3.0 * st["x2"].double()
        return torch.sigmoid(lin) if case["sigmoid"] else lin
    if op in ("join", "join_part"):
        return _exact_join(case, seed)
    if op in ("sort", "sort_msb"):
        keys, order = torch.sort(_sort_keys(case, seed), stable=True)
        return keys, order.to(torch.int32)
    if op == "query":
        return _exact_query(case, seed)
    return _exact_star(case, seed)
