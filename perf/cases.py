"""The queries this engine is measured on, each through the Python binding's public calls.

Every case evaluates the engine's query shape,

    SELECT g, SUM(..), SUM(price * (100 - disc)), COUNT(*), AVG(..)
    FROM fact JOIN dim ON fk = pk [JOIN dim2 ..] WHERE date BETWEEN .. GROUP BY g

on synthetic star-schema tables made on the GPU from the seed: a day column over seven years (2,557 days), two- and
three-valued flags, decimal money as scaled int64, foreign keys uniform or Zipf(0.8) over the dimension's rows.
Kinds of case:

  star    few groups (flag, status, a dimension attribute; 150 groups, 600 with a second dimension); the caller
          reads the small result on the host
  orders  many groups (by an order or account id of the fact table); the result stays on the device
  batch   several uneven queries captured into one launch; results stay on the device
  paged   the star query on tables in page-locked host pages, streamed through the prefetch ring
  spill   the same with a build side larger than the device budget: partitioned, most partitions spilled
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2508_05029_gb300 import theseus as T

DAYS = 2557
CUTOFF_98 = 2504          # date <= 2504 keeps 97.97% of uniform days
I64_MIN = -(1 << 63)
DEV = "cuda"


# ------------------------------------------------------------------ the cases

def _star(name, n, n_dim, keys="dense", skew="uniform", cutoff=CUTOFF_98, repeat=1, wide=False, n_dim2=0):
    return dict(name=name, kind="star", n=n, n_dim=n_dim, keys=keys, skew=skew, cutoff=cutoff, repeat=repeat,
                wide=wide, n_dim2=n_dim2)


def _orders(name, n, n_dim, n_keys, ids="dense", adjacent=True, days=CUTOFF_98 + 1):
    return dict(name=name, kind="orders", n=n, n_dim=n_dim, n_keys=n_keys, ids=ids, adjacent=adjacent, days=days)


def listed():
    return [
        # the smallest request a served dashboard sends: nearly all of it is launches, allocation and the read back
        _star("star_10k", 10_007, 1_000),
        # one device-resident batch of the paper's size joined to a small dimension
        _star("star_1m", 1_000_000, 10_000),
        # the headline query: a 60M-row fact table, skewed foreign keys, a dense-keyed 2M-row dimension
        _star("star_60m", 60_000_000, 2_000_000, skew="zipf"),
        # the same when the dimension's keys are sparse 64-bit ids, so the join needs a hashed table
        _star("star_sparse_60m", 60_000_000, 2_000_000, keys="sparse", skew="zipf"),
        # a star join with a second, large dimension whose own predicate keeps 12% of it (lookahead filter)
        _star("star_two_dims_60m", 60_000_000, 2_000_000, skew="zipf", n_dim2=32_000_000),
        # a join that fans out (three dimension rows per key) over money wide enough that sums leave 64 bits
        _star("star_fanout_wide_20m", 20_000_003, 1_500_000, keys="sparse", repeat=3, wide=True),
        # totals per order for 26 days of seven years: a 1% filter ahead of many groups
        _orders("orders_26_days_60m", 60_000_000, 2_000_000, 15_000_000, days=26),
        # totals per order over nearly all rows: 15M groups, the lines of an order next to each other
        _orders("orders_60m", 60_000_000, 2_000_000, 15_000_000),
        # totals per account, account ids sparse in 40 bits and in no order: a hashed aggregation
        _orders("accounts_30m", 30_000_001, 500_000, 3_000_000, ids="sparse", adjacent=False),
        # twelve uneven queries of a dashboard in one captured launch
        dict(name="batch_12", kind="batch", queries=12, median=500_000, sizes=7),
        # the star query on tables in host pages: bit-packed columns copied, widened and aggregated in a pipeline
        dict(name="paged_12m", kind="paged", n=12_000_000, n_dim=500_000),
        # a build side larger than the device budget: the hybrid join partitions, spills and reads back
        dict(name="spill_8m", kind="spill", n=8_000_000, n_dim=3_000_000, partitions=16),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["star", "star", "star", "orders", "orders", "orders", "batch", "paged", "spill"])
    if kind == "star":
        two = rng.random() < 0.25
        repeat = rng.choice([1, 1, 1, 2, 3])
        least = 200_000 if two else 6_000   # passing rows: every one of the groups keeps some
        n = max(size(10_000, 60_000_000 if repeat == 1 else 20_000_003), 2 * least if two else 10_000)
        c = _star("", n, size(1_000, 2_000_000), keys=rng.choice(["dense", "sparse"]),
                  skew=rng.choice(["uniform", "zipf"]), cutoff=rng.randrange(max(50, DAYS * least // n), DAYS),
                  repeat=repeat, wide=rng.random() < 0.25, n_dim2=size(50_000, 32_000_000) if two else 0)
    elif kind == "orders":
        n = size(100_000, 60_000_000)
        ids = rng.choice(["dense", "sparse"])
        if ids == "sparse":
            n = min(n, 30_000_001)
        c = _orders("", n, size(1_000, 2_000_000), max(5_000, int(n / rng.uniform(2, 40))), ids=ids,
                    adjacent=rng.random() < 0.5, days=rng.choice([rng.randrange(20, 200), rng.randrange(700, DAYS)]))
    elif kind == "batch":
        c = dict(kind=kind, queries=rng.randrange(3, 13), median=size(100_000, 500_000), sizes=rng.randrange(1000))
    elif kind == "paged":
        c = dict(kind=kind, n=size(100_000, 12_000_000), n_dim=size(1_000, 500_000))
    else:
        c = dict(kind=kind, n=size(1_000_000, 8_000_000), n_dim=size(1_000_000, 3_000_000),
                 partitions=rng.choice([8, 16, 32, 64]))
    c.pop("name", None)
    return c


def _batch_sizes(case):
    """Per query (fact rows, dimension rows, groups, cutoff): lognormal facts, log-uniform dimensions and groups."""
    r = random.Random(case["sizes"])
    out = []
    for _ in range(case["queries"]):
        n = int(min(max(case["median"] * math.exp(1.5 * r.gauss(0, 1)), 10_000), 10_000_000))
        out.append((n, int(math.exp(r.uniform(math.log(1e3), math.log(1e6)))),
                    int(math.exp(r.uniform(math.log(4), math.log(1e5)))), r.randrange(100, DAYS)))
    return out


# ----------------------------------------------------------------------- data

def _mix(i):
    """A bijection of int64 (distinct inputs give distinct sparse keys)."""
    i = i * -7046029254386353131 + 0x1234567
    i = i ^ ((i >> 31) & 0x1FFFFFFFF)
    i = i * -4658895280553007687
    return i ^ ((i >> 29) & 0x7FFFFFFFF)


def _rand(g, lo, hi, n, dtype=torch.int64):
    return torch.randint(lo, hi + 1, (n,), generator=g, device=DEV, dtype=dtype)


def _ref_rows(g, n, n_keys, skew):
    """Which of the n_keys dimension keys each fact row refers to."""
    if skew == "uniform":
        return _rand(g, 0, n_keys - 1, n)
    cdf = torch.cumsum(torch.arange(1, n_keys + 1, device=DEV, dtype=torch.float64).pow_(-0.8), 0)
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * cdf[-1]
    return torch.searchsorted(cdf, u).clamp_(max=n_keys - 1)


def _measures(g, n, wide=False):
    price = (90_000, 10_500_000) if not wide else (-9_000_000_000_000_000, 90_000_000_000_000_000)
    return dict(date=_rand(g, 0, DAYS - 1, n, torch.int32), qty=_rand(g, 1, 50, n) * 100, price=_rand(g, *price, n),
                disc=_rand(g, 0, 10, n), flag=_rand(g, 0, 2, n, torch.uint8), status=_rand(g, 0, 1, n, torch.uint8))


def _dim(g, n_dim, keys, repeat=1):
    """A dimension of unique scrambled keys (each on `repeat` rows); pk of key k is at rows k * repeat .."""
    n_keys = max(1, n_dim // repeat)
    if keys == "dense":
        pk = torch.randperm(n_keys, generator=g, device=DEV).to(torch.int32)
    else:
        pk = _mix(torch.arange(n_keys, device=DEV) + int(_rand(g, 0, 1 << 40, 1)))
    return dict(pk=pk.repeat_interleave(repeat), attr=_rand(g, 0, 24, n_keys * repeat, torch.int32)), pk


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _star_data(case, seed):
    """Fact and dimension columns, and the dimension key each fact row refers to (per dimension)."""
    g = _gen(seed)
    n = case["n"]
    dim, pk = _dim(g, case["n_dim"], case.get("keys", "dense"), repeat=case.get("repeat", 1))
    ref = _ref_rows(g, n, len(pk), case.get("skew", "uniform"))
    fact = dict(fk=pk[ref], **_measures(g, n, case.get("wide", False)))
    dim2 = ref2 = None
    if case.get("n_dim2"):
        dim2, pk2 = _dim(g, case["n_dim2"], "sparse")
        dim2["band"] = _rand(g, 0, 3, case["n_dim2"], torch.uint8)
        ref2 = _rand(g, 0, case["n_dim2"] - 1, n)
        fact["fk2"] = pk2[ref2]
    return fact, dim, ref, dim2, ref2


def _orders_data(case, seed):
    """Which rows belong to the same order and pass the filter is the case's own (so is the number of groups); the
    ids, keys and money are the seed's."""
    g, own = _gen(seed), _gen(case["n"])
    n, k = case["n"], case["n_keys"]
    dim, pk = _dim(g, case["n_dim"], "dense")
    ref = _ref_rows(g, n, len(pk), "uniform")
    ids = torch.randperm(k, generator=g, device=DEV)
    if case["ids"] == "sparse":
        ids = (ids * 0x9E3779B97B) & ((1 << 40) - 1)   # an odd multiplier: distinct
        ids = ids ^ (ids >> 17)
    at = torch.arange(n, device=DEV) * k // n if case["adjacent"] else _rand(own, 0, k - 1, n)
    date = _rand(own, 0, DAYS - 1, n, torch.int32)
    m = _measures(g, n)
    return dict(fk=pk[ref], date=date, price=m["price"], disc=m["disc"], okey=ids[at]), dim


def _batch_data(case, seed):
    """Days, attributes and references are the case's own (and with them each query's number of groups)."""
    out = []
    for i, (n, n_dim, groups, cutoff) in enumerate(_batch_sizes(case)):
        g, own = _gen(seed * 64 + i), _gen(case["sizes"] * 64 + i)
        dim, pk = _dim(g, n_dim, "dense")
        dim["attr"] = _rand(own, 0, groups - 1, n_dim, torch.int32)
        ref = _rand(own, 0, n_dim - 1, n)
        m = _measures(g, n)
        date = _rand(own, 0, DAYS - 1, n, torch.int32)
        out.append((dict(fk=pk[ref], date=date, qty=m["qty"], price=m["price"], disc=m["disc"]), dim, ref))
    return out


# -------------------------------------------------------------------- queries

_AGGS = [("sum", "qty"), ("sum_mul_sub", "price", 100, "disc"), ("count",), ("avg", "disc")]


def _star_query(case):
    q = dict(filter=dict(col="date", lo=I64_MIN, hi=case.get("cutoff", CUTOFF_98)),
             join=dict(fact_col="fk", dim_col="pk", many=case.get("repeat", 1) > 1),
             group=[("fact", "flag", 2), ("fact", "status", 1), ("dim", "attr", 5)], aggs=_AGGS)
    if case.get("n_dim2"):
        q["group"] = q["group"] + [("dim1", "band", 2)]
        q["extra_joins"] = [dict(fact_col="fk2", dim_col="pk", dim_filter=dict(col="attr", lo=0, hi=2))]
    return q


def _orders_lo(case):
    return 0 if case["days"] > DAYS // 2 else (DAYS - case["days"]) // 3


def _orders_query(case):
    lo = _orders_lo(case)
    return dict(filter=dict(col="date", lo=lo, hi=lo + case["days"] - 1), join=dict(fact_col="fk", dim_col="pk"),
                group=[("fact", "okey", 64)], aggs=[("sum_mul_sub", "price", 100, "disc"), ("count",)])


def _batch_query(groups, cutoff):
    return dict(filter=dict(col="date", lo=I64_MIN, hi=cutoff), join=dict(fact_col="fk", dim_col="pk"),
                group=[("dim", "attr", max(1, (groups - 1).bit_length()))], aggs=_AGGS)


# --------------------------------------------------------------------- states

_engines = {}
PAGED_BATCH = 1 << 20
SPILL_BATCH = 250_000


def _engine(kind):
    """One engine per way of holding data, as a program keeps one: device tables, host pages, a small budget."""
    if kind not in _engines:
        if kind == "paged":
            _engines[kind] = T.Engine(page_bytes=8 << 20, n_pages=192, batch_rows=PAGED_BATCH)
        elif kind == "spill":
            _engines[kind] = T.Engine(page_bytes=2 << 20, n_pages=768, batch_rows=SPILL_BATCH)
        else:
            _engines[kind] = T.Engine()
    return _engines[kind]


class _State:
    """Tables, plans and the last result of one prepared case; gives them back when it goes."""

    def __init__(self, case):
        self.case, self.tables, self.plans, self.batch = case, [], [], None

    def __del__(self):
        if self.batch is not None:
            self.batch.destroy()
        for p in self.plans:
            p.destroy()
        for t in self.tables:
            t.destroy()


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    eng = _engine(kind)
    if kind == "batch":
        for (fact, dim, _), (_, _, groups, cutoff) in zip(_batch_data(case, seed), _batch_sizes(case)):
            torch.cuda.synchronize()
            ft, dt = eng.table_from_torch(fact), eng.table_from_torch(dim)
            s.tables += [ft, dt]
            s.plans.append(eng.plan(ft, dt, _batch_query(groups, cutoff)))
        s.batch = T.Batch(eng, s.plans)
        return s
    extra, dim2 = {}, None
    if kind == "orders":
        fact, dim = _orders_data(case, seed)
        query = _orders_query(case)
    else:
        fact, dim, _, dim2, _ = _star_data(_as_star(case), seed)
        query = _star_query(_as_star(case))
    torch.cuda.synchronize()
    if kind in ("paged", "spill"):
        tabs = [eng.table_from_numpy({k: v.cpu().numpy() for k, v in t.items()}) for t in (fact, dim)]
    else:
        tabs = [eng.table_from_torch(t) for t in (fact, dim)]
    s.tables += tabs
    if dim2 is not None:
        s.tables.append(eng.table_from_torch(dim2))
        extra["extra_dims"] = [s.tables[-1]]
    if kind == "spill":
        extra["join_partitions"] = case["partitions"]
        # the streaming buffers and about a third of the build side's table
        s.budget = (100 << 20) + case["n_dim"] * 12
    s.plans.append(eng.plan(tabs[0], tabs[1], query, **extra))
    return s


def _as_star(case):
    """paged and spill cases run the star query; spill joins on sparse 64-bit keys."""
    if case["kind"] == "star":
        return case
    return _star("", case["n"], case["n_dim"], keys="sparse" if case["kind"] == "spill" else "dense")


class _View:
    """Device memory of a result as an array torch can read in place; keeps the result alive."""

    def __init__(self, owner, ptr, shape, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = dict(shape=shape, typestr=typestr, data=(ptr, False), version=3)


class _Owner:
    def __init__(self, res):
        self.res = res

    def __del__(self):
        self.res.free()


def _device_outputs(res, aggs, owner):
    """The whole result as tensors on its own device memory, which owner holds."""
    n = res.n_groups

    def view(ptr, shape, typestr="<i8"):
        if n == 0:
            return torch.empty(shape, device=DEV, dtype=torch.float64 if typestr == "<f8" else torch.int64)
        return torch.as_tensor(_View(owner, ptr, shape, typestr), device=DEV)

    out = dict(keys=view(T.tp_result_device_keys(res.h), (n,)), counts=view(T.tp_result_device_count(res.h), (n,)))
    for a, ag in enumerate(aggs):
        if ag[0] == "avg":
            out["avg%d" % a] = view(T.tp_result_device_avg(res.h, a), (n,), "<f8")
        elif ag[0] != "count":
            out["sum%d" % a] = view(T.tp_result_device_sum(res.h, a), (n, 2))
    return out


def _host_outputs(res, aggs):
    with res:
        out = dict(keys=res.keys(), counts=res.counts())
        for a, ag in enumerate(aggs):
            if ag[0] == "avg":
                out["avg%d" % a] = res.avg(a)
            elif ag[0] != "count":
                out["sum%d" % a] = res.sum_words(a)
    return {k: v.view(np.int64) if v.dtype == np.uint64 else v for k, v in out.items()}


def run(state):
    kind = state.case["kind"]
    if kind == "batch":
        res = state.batch.execute()   # valid until the next execute, owned by the batch
        return [_device_outputs(r, p.aggs, state) for r, p in zip(res, state.plans)]
    plan = state.plans[0]
    if kind == "spill":
        plan.eng.set_budget(state.budget)
    res = plan.execute()
    return _device_outputs(res, plan.aggs, _Owner(res)) if kind == "orders" else _host_outputs(res, plan.aggs)


# ------------------------------------------------------- what a pass must move

def work(case):
    """Each column a query reads once at its width, and each result row once.  Under a selective filter the other
    columns count for the passing rows.  Host pages hold bit-packed columns: their packed widths."""
    kind = case["kind"]
    if kind == "batch":
        b = sum(n * (4 + 4 + 24) + d * 8 + g * 56 for n, d, g, _ in _batch_sizes(case))
        return dict(bytes=b, flops=0)
    if kind == "orders":
        n, share = case["n"], min(1.0, case["days"] / DAYS)
        groups = case["n_keys"] * (1 - (1 - share) ** (n / case["n_keys"]))
        rest = n * share if share < 0.25 else n
        return dict(bytes=int(n * 4 + rest * 28 + case["n_dim"] * 8 + groups * 32), flops=0)
    if kind == "paged":
        fk = max(1, (case["n_dim"] - 1).bit_length())
        return dict(bytes=int(case["n"] * (fk + 12 + 13 + 24 + 4 + 2 + 1) / 8 + case["n_dim"] * (fk + 5) / 8), flops=0)
    if kind == "spill":
        return dict(bytes=case["n"] * 38 + case["n_dim"] * 12, flops=0)
    k = 8 if case["keys"] == "sparse" else 4
    b = case["n"] * (30 + k) + case["n_dim"] * (k + 4)
    if case["n_dim2"]:
        b += case["n"] * 8 + case["n_dim2"] * 13
    return dict(bytes=b, flops=0)


# ---------------------------------------------------- the same in plain torch

def _group(key, terms):
    """keys ascending, counts, and per term the exact sum as (low word, high word)."""
    keys, inv = torch.unique(key, return_inverse=True)
    counts = torch.zeros(len(keys), device=DEV, dtype=torch.int64).index_add_(0, inv, torch.ones_like(inv))
    sums = []
    for t in terms:
        # two 32-bit halves cannot overflow a 64-bit sum; then carry into the high word
        lo = torch.zeros(len(keys), device=DEV, dtype=torch.int64).index_add_(0, inv, t & 0xFFFFFFFF)
        hi = torch.zeros(len(keys), device=DEV, dtype=torch.int64).index_add_(0, inv, t >> 32)
        hi += lo >> 32
        sums.append(torch.stack([(hi << 32) | (lo & 0xFFFFFFFF), hi >> 32], 1))
    return keys, counts, sums


def _few_groups(key, f):
    keys, counts, (qty, money, disc) = _group(key, [f["qty"], f["price"] * (100 - f["disc"]), f["disc"]])
    return dict(keys=keys, counts=counts, sum0=qty, sum1=money, avg3=disc[:, 0].double() / counts.double())


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for (f, dim, ref), (_, _, _, cutoff) in zip(_batch_data(case, seed), _batch_sizes(case)):
            keep = f["date"] <= cutoff
            out.append(_few_groups(dim["attr"][ref[keep]].long(), {k: v[keep] for k, v in f.items()}))
        return out
    if kind == "orders":
        f, _ = _orders_data(case, seed)
        lo = _orders_lo(case)
        keep = (f["date"] >= lo) & (f["date"] < lo + case["days"])
        keys, counts, (money,) = _group(f["okey"][keep], [(f["price"] * (100 - f["disc"]))[keep]])
        return dict(keys=keys, counts=counts, sum0=money)
    c = _as_star(case)
    f, dim, ref, dim2, ref2 = _star_data(c, seed)
    keep = f["date"] <= c["cutoff"]
    if dim2 is not None:
        keep &= dim2["attr"][ref2] <= 2
    f, ref = {k: v[keep] for k, v in f.items()}, ref[keep]
    key = f["flag"].long() * 2 + f["status"].long()
    attr = dim["attr"].view(-1, c["repeat"])
    keys = [key * 32 + attr[ref, m] for m in range(c["repeat"])]
    if dim2 is not None:
        band = dim2["band"][ref2[keep]].long()
        keys = [k * 4 + band for k in keys]
    return _few_groups(torch.cat(keys), {k: v.repeat(c["repeat"]) for k, v in f.items()})
