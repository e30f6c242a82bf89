"""Fan-out joins whose sums pass a bound only because every fact row counts once
per partner: 32-bit words of a CTA's table, int64 sums of few and of many
groups, and build rows that change between two executions of one plan; count,
sums and averages against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2508_05029_gb300 import theseus as T
from tests.helpers import assert_matches_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_05029_gb300 import build
    build.build()


def _up(e, cols):
    import torch
    dev = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in cols.items()}
    t = e.table_from_torch(dev)
    torch.cuda.synchronize()
    return t, dev


def _check(fact, dim, q, flags=0):
    e = T.Engine(flags=flags)
    try:
        ft, _ = _up(e, fact)
        dt, _ = _up(e, dim)
        p = e.plan(ft, dt, q)
        ref = oracle.run_query(fact, dim, q)
        for _ in range(2):   # the build rows of a key counted first, then checked
            with p.execute() as r:
                assert_matches_oracle(r, ref, q["aggs"])
        return e.stats()
    finally:
        e.close()


FLAGS = [0, T.TP_FLAG_NO_JIT, T.TP_FLAG_NO_DIRECT_JOIN]


@pytest.mark.parametrize("flags", FLAGS)
@pytest.mark.parametrize("wide", [True, False])
@pytest.mark.parametrize("fan", [1, 3, 16])
def test_terms_of_a_cta_pass_32_bits(fan, wide, flags):
    """A CTA's rows times the terms stay just below 2^32, times the partners they
    do not (7,744 rows of a CTA on 152 SMs times 500,000)."""
    rng = np.random.default_rng(fan)
    n, m = 1_000_000, 50_000
    i64 = np.iinfo(np.int64)
    fact = dict(fk=rng.integers(0, m, n).astype(np.int32), v=rng.integers(0, 500_000, n, endpoint=True),
                w=rng.integers(i64.min, i64.max, n, endpoint=True), d=rng.integers(0, 1 << 40, n, endpoint=True))
    dim = dict(pk=np.repeat(np.arange(m, dtype=np.int32), fan), attr=np.zeros(m * fan, np.int32))
    aggs = [("sum", "v"), ("count",), ("avg", "v"), ("sum", "d")] + ([("sum", "w"), ("avg", "w")] if wide else [])
    q = dict(filter=None, join=dict(fact_col="fk", dim_col="pk", many=True), group=[("dim", "attr", 3)], aggs=aggs)
    _check(fact, dim, q, flags)


@pytest.mark.parametrize("flags", FLAGS)
@pytest.mark.parametrize("key_bits", [3, 20])
def test_sums_leave_int64_through_their_partners(key_bits, flags):
    """Sums of 2^62 before the join, 2^65 after it; few groups and many."""
    rng = np.random.default_rng(key_bits)
    n, m, fan = 4_096, 64, 8
    fact = dict(fk=rng.integers(0, m, n), key=np.where(rng.random(n) < 0.9, 5, rng.integers(0, 1 << key_bits, n)),
                v=np.full(n, 1 << 50), s=np.full(n, -(1 << 50)))
    dim = dict(pk=np.repeat(np.arange(m) * 1_000_003, fan))
    fact["fk"] = fact["fk"] * 1_000_003
    q = dict(filter=None, join=dict(fact_col="fk", dim_col="pk", many=True), group=[("fact", "key", key_bits)],
             aggs=[("sum", "v"), ("avg", "v"), ("sum", "s"), ("count",)])
    _check(fact, dim, q, flags)


def test_build_rows_that_gain_partners_between_executions():
    rng = np.random.default_rng(9)
    n, m = 300_000, 40_000
    fact = dict(fk=rng.integers(0, m // 8, n).astype(np.int32), v=rng.integers(0, 1_200_000, n, endpoint=True))
    dim = dict(pk=np.arange(m, dtype=np.int32), attr=np.zeros(m, np.int32))
    q = dict(filter=None, join=dict(fact_col="fk", dim_col="pk", many=True), group=[("dim", "attr", 3)],
             aggs=[("sum", "v"), ("count",), ("avg", "v")])
    e = T.Engine()
    try:
        ft, _ = _up(e, fact)
        dt, dev = _up(e, dim)
        p = e.plan(ft, dt, q)
        with p.execute() as r:
            assert_matches_oracle(r, oracle.run_query(fact, dim, q), q["aggs"])
        import torch
        dim["pk"][: m - 2] //= 8          # eight rows per key; the column's bounds stay what they were
        dev["pk"].copy_(torch.from_numpy(dim["pk"]).cuda())
        torch.cuda.synchronize()
        ref = oracle.run_query(fact, dim, q)
        for retries in (1, 1):
            with p.execute() as r:
                assert_matches_oracle(r, ref, q["aggs"])
            assert e.stats()["retries"] == retries
    finally:
        e.close()
