"""Many-group aggregation through partitioned records: dense key ranges and
sparse ones, rows of a key next to each other or in no order, clustered keys,
one hot key (a partition overflows and the query falls back), selective
filters, zero to four sums, ragged sizes; against the oracle bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_05029_gb300 import theseus as T
from tests.helpers import assert_matches_oracle

pytestmark = pytest.mark.gpu
ROWS = (4 << 20)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_05029_gb300 import build
    build.build()


def _keys(rng, kind, n, groups):
    if kind == "adjacent":
        return (rng.permutation(groups) + 1_000_003)[np.arange(n) * groups // n]
    if kind == "shuffled":
        return rng.integers(0, groups, n) + 7
    if kind == "ascending":
        return np.arange(n, dtype=np.int64) * groups // n
    if kind == "sparse":
        return (rng.permutation(groups).astype(np.int64) * 0x9E3779B97B & ((1 << 40) - 1))[rng.integers(0, groups, n)]
    if kind == "sparse-clustered":   # runs of consecutive ids, far apart: a few ordering buckets hold many keys
        return (np.arange(groups, dtype=np.int64) % 97 + (np.arange(groups, dtype=np.int64) // 97 << 21))[
            rng.integers(0, groups, n)]
    if kind == "hot":                # too small a share for the sample to see, too large for a partition
        k = rng.integers(0, groups, n)
        k[rng.integers(0, n, n // 300)] = 12345
        return k
    return np.where(rng.random(n) < 0.5, 5, rng.integers(0, groups, n))   # "half": one key has half the rows


def _run(fact, dim, q, flags=0, **kw):
    e = T.Engine(flags=flags)
    try:
        up = lambda t: e.table_from_torch({k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in t.items()})
        ft, dt = up(fact), up(dim) if dim else None
        torch.cuda.synchronize()
        p = e.plan(ft, dt, q, **kw)
        ref = oracle.run_query(fact, dim, q)
        for _ in range(2):   # sampled, then from the plan's history
            with p.execute() as r:
                assert_matches_oracle(r, ref, q["aggs"])
        return e.stats()
    finally:
        e.close()


@pytest.mark.parametrize("kind,groups", [("adjacent", 1_048_576), ("shuffled", 300_000), ("shuffled", 3_000_000),
                                         ("ascending", 1_500_001), ("sparse", 400_000), ("sparse", 2_500_000),
                                         ("sparse-clustered", 500_000), ("hot", 2_000_000), ("half", 2_000_000)])
@pytest.mark.parametrize("sel", [1.0, 0.03])
def test_key_distributions(kind, groups, sel):
    rng = np.random.default_rng(groups)
    n = ROWS + 2049
    fact = dict(key=_keys(rng, kind, n, groups).astype(np.int64), d=rng.integers(0, 1000, n).astype(np.int32),
                fk=rng.integers(0, 5000, n).astype(np.int32), a=rng.integers(-10**9, 10**9, n))
    dim = dict(pk=np.arange(100, 4900, dtype=np.int32))
    q = dict(filter=dict(col="d", lo=0, hi=int(1000 * sel) - 1), join=dict(fact_col="fk", dim_col="pk"),
             group=[("fact", "key", 64)], aggs=[("sum", "a"), ("count",), ("avg", "a")])
    _run(fact, dim, q)


@pytest.mark.parametrize("aggs", [[("count",)], [("sum", "a")], [("sum", "a"), ("sum_mul_sub", "a", 7, "u")],
                                  [("sum", "a"), ("avg", "u"), ("sum_mul_sub", "a", -3, "w"), ("avg", "w")],
                                  [("sum", "a")] * 5])
@pytest.mark.parametrize("tail", [0, 1, 3, 2047])
def test_sums_and_tails(aggs, tail):
    rng = np.random.default_rng(tail)
    n = ROWS + tail
    fact = dict(hi=rng.integers(0, 900, n).astype(np.int32), lo=rng.integers(0, 1000, n).astype(np.int64),
                a=rng.integers(-10**6, 10**6, n), u=rng.integers(0, 255, n).astype(np.uint8),
                w=rng.integers(-500, 500, n).astype(np.int32))
    q = dict(filter=None, join=None, group=[("fact", "hi", 10), ("fact", "lo", 10)], aggs=aggs)
    _run(fact, None, q)


def test_a_field_beyond_its_bits_is_refused():
    n = ROWS
    fact = dict(k=np.arange(n, dtype=np.int64), a=np.ones(n, np.int64))
    fact["k"][17] = 1 << 30
    q = dict(filter=None, join=None, group=[("fact", "k", 24)], aggs=[("sum", "a")])
    with pytest.raises(T.TPError) as err:
        _run_gpu_only(fact, q)
    assert err.value.code == T.TP_E_RANGE


def _run_gpu_only(fact, q):
    e = T.Engine()
    try:
        ft = e.table_from_torch({k: torch.from_numpy(v).cuda() for k, v in fact.items()})
        torch.cuda.synchronize()
        e.plan(ft, None, q).execute().free()
    finally:
        e.close()
