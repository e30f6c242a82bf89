"""Every way into the partitioned records: compiled and ahead-of-time scans, of all
rows and of selected ones, joined through direct, packed, unpacked and 32-bit
tables, zero to four sums and ragged tails; keys outside the bounds that were
taken and a refused reservation fall back.  Against the oracle bit for bit, and
what ran is checked: a record aggregation is one compiled launch, or with
TP_FLAG_NO_JIT as many launches as the compiled one takes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_05029_gb300 import theseus as T
from tests.helpers import assert_matches_oracle

pytestmark = pytest.mark.gpu
ROWS = 4 << 20
GROUPS = 300_000


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_05029_gb300 import build
    build.build()


def _up(e, cols):
    t = e.table_from_torch({k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in cols.items()})
    torch.cuda.synchronize()
    return t


def _launches(fact, dim, q, flags, **kw):
    """(compiled launches, launches) of a second execution; both are checked."""
    e = T.Engine(flags=flags)
    try:
        ft, dt = _up(e, fact), _up(e, dim) if dim else None
        p = e.plan(ft, dt, q, expected_groups=GROUPS, **kw)
        ref = oracle.run_query(fact, dim, q)
        for _ in range(2):
            s0 = e.stats()
            with p.execute() as r:
                assert_matches_oracle(r, ref, q["aggs"])
            s1 = e.stats()
        assert s1["retries"] == 0
        return s1["jit_launches"] - s0["jit_launches"], s1["kernel_launches"] - s0["kernel_launches"]
    finally:
        e.close()


def _both(fact, dim, q, flags=0, **kw):
    jit, n = _launches(fact, dim, q, flags, **kw)
    assert jit == 1
    assert _launches(fact, dim, q, flags | T.TP_FLAG_NO_JIT, **kw) == (0, n)


JOINS = {   # key values of m dimension rows, key type, flags: the table that serves them
    "none": None,
    "direct": (lambda rng, m: np.arange(100, 100 + m), np.int32, 0),
    "packed": (lambda rng, m: rng.permutation(m) * 0x9E3779B97B - 5, np.int64, 0),
    "hash32": (lambda rng, m: rng.permutation(m) * 401 - 7, np.int32, 0),
    "unpacked": (lambda rng, m: rng.permutation(m) * 0x9E3779B97B - 5, np.int64, "0.9"),
}


@pytest.mark.parametrize("join", list(JOINS))
@pytest.mark.parametrize("sel", [1.0, 0.2])
@pytest.mark.parametrize("ids", ["dense", "sparse"])
def test_scans_and_joins(join, sel, ids):
    rng = np.random.default_rng(len(join) + int(10 * sel))
    n, m = ROWS + 2049, 6_000
    k = rng.integers(0, GROUPS, n)
    fact = dict(key=k + 7 if ids == "dense" else k * 0x9E3779B9 & ((1 << 40) - 1),
                d=rng.integers(0, 1000, n).astype(np.int32), a=rng.integers(-10**9, 10**9, n))
    fact["key"] = fact["key"].astype(np.int64)
    q = dict(filter=None if sel == 1.0 else dict(col="d", lo=0, hi=int(1000 * sel) - 1), join=None,
             group=[("fact", "key", 64)], aggs=[("sum", "a"), ("count",), ("avg", "a")])
    dim, kw = None, {}
    if JOINS[join]:
        keys, dt, opt = JOINS[join]
        pk = keys(rng, m).astype(dt)
        dim = dict(pk=pk[: m - 1000])          # some fact rows have no partner
        fact["fk"] = rng.choice(pk, n)
        q["join"] = dict(fact_col="fk", dim_col="pk")
        if opt:
            kw["load_factor"] = float(opt)     # fuller than what packs
    _both(fact, dim, q, **kw)


@pytest.mark.parametrize("aggs", [[("count",)], [("avg", "u")], [("sum", "a"), ("sum_mul_sub", "a", 7, "u")],
                                  [("sum", "a"), ("avg", "u"), ("sum_mul_sub", "a", -3, "w")],
                                  [("sum", "a"), ("avg", "u"), ("sum_mul_sub", "a", -3, "w"), ("avg", "w")]])
@pytest.mark.parametrize("tail,sel", [(0, 0.2), (1, 1.0), (3, 0.2), (2047, 1.0)])
def test_sums_and_tails(aggs, tail, sel):
    rng = np.random.default_rng(tail)
    n = ROWS + tail
    fact = dict(hi=rng.integers(0, 900, n).astype(np.int32), lo=rng.integers(0, 1000, n).astype(np.int64),
                d=rng.integers(0, 200, n).astype(np.uint8), a=rng.integers(-10**6, 10**6, n),
                u=rng.integers(0, 255, n).astype(np.uint8), w=rng.integers(-500, 500, n).astype(np.int32))
    q = dict(filter=None if sel == 1.0 else dict(col="d", lo=10, hi=9 + int(200 * sel)), join=None,
             group=[("fact", "hi", 10), ("fact", "lo", 10)], aggs=aggs)
    _both(fact, None, q)


@pytest.mark.parametrize("flags", [0, T.TP_FLAG_NO_JIT])
def test_a_key_outside_the_bounds_falls_back(flags):
    """A caller writes keys into a registered column that its bounds do not cover."""
    rng = np.random.default_rng(11)
    n = ROWS + 5
    fact = dict(key=rng.integers(0, GROUPS, n) * 5_000_011, a=rng.integers(0, 1000, n))
    q = dict(filter=None, join=None, group=[("fact", "key", 64)], aggs=[("sum", "a"), ("count",)])
    e = T.Engine(flags=flags)
    try:
        dev = {k: torch.from_numpy(v).cuda() for k, v in fact.items()}
        ft = e.table_from_torch(dev)
        torch.cuda.synchronize()
        p = e.plan(ft, None, q, expected_groups=GROUPS)
        for retries in (0, 1, 1):
            with p.execute() as r:
                assert_matches_oracle(r, oracle.run_query(fact, None, q), q["aggs"])
            assert e.stats()["retries"] == retries
            fact["key"][n // 2] = 1 << 62
            dev["key"][n // 2] = 1 << 62
            torch.cuda.synchronize()
    finally:
        e.close()


@pytest.mark.parametrize("flags", [0, T.TP_FLAG_NO_JIT])
def test_a_refused_reservation_falls_back(flags):
    """The records take about 90 MB beside the result, the table 32 MB."""
    rng = np.random.default_rng(12)
    fact = dict(key=rng.integers(0, GROUPS, ROWS) * 5_000_011, a=rng.integers(0, 1000, ROWS))
    q = dict(filter=None, join=None, group=[("fact", "key", 64)], aggs=[("sum", "a"), ("count",)])
    e = T.Engine(flags=flags, device_budget_bytes=80 << 20)
    try:
        ft = _up(e, fact)
        p = e.plan(ft, None, q, expected_groups=GROUPS)
        ref = oracle.run_query(fact, None, q)
        for budget, jit in ((80 << 20, 0), (200 << 20, 0 if flags else 1)):
            e.set_budget(budget)
            s0 = e.stats()["jit_launches"]
            with p.execute() as r:
                assert_matches_oracle(r, ref, q["aggs"])
            assert e.stats()["jit_launches"] - s0 == jit
            assert e.stats()["peak_reserved"] <= budget
    finally:
        e.close()
