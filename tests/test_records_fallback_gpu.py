"""Many-group aggregation when its records cannot be had or did not suit the
plan: the query runs through the global table, and a later execution takes the
records again.  A record scan is a run-time compiled launch, the global table's
kernels are not."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_05029_gb300 import theseus as T
from tests.helpers import assert_matches_oracle

pytestmark = pytest.mark.gpu
ROWS = (4 << 20) + 1025
MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_05029_gb300 import build
    build.build()


class Case:
    """A plan over rows of (key, a); each run is checked and says what it launched."""

    def __init__(self, fact, q, **kw):
        self.fact, self.q, self.e = fact, q, T.Engine(**kw)
        self.dev = {k: torch.from_numpy(v).cuda() for k, v in fact.items()}
        self.table = self.e.table_from_torch(self.dev)
        torch.cuda.synchronize()
        self.plan = self.e.plan(self.table, None, q)
        self.ref = oracle.run_query(fact, None, q)

    def change(self, key):
        self.fact["key"][:] = key
        self.dev["key"].copy_(torch.from_numpy(key).cuda())
        torch.cuda.synchronize()
        self.ref = oracle.run_query(self.fact, None, self.q)

    def run(self):
        """(record scans, retries) of one execution"""
        s0 = self.e.stats()
        with self.plan.execute() as r:
            assert_matches_oracle(r, self.ref, self.q["aggs"])
        s1 = self.e.stats()
        return s1["jit_launches"] - s0["jit_launches"], s1["retries"] - s0["retries"]


def _query(flt=None):
    return dict(filter=flt, join=None, group=[("fact", "key", 64)], aggs=[("sum", "a"), ("count",)])


def _fact(key, seed=1):
    return dict(key=np.ascontiguousarray(key, np.int64), a=np.random.default_rng(seed).integers(-10**9, 10**9, len(key)))


@pytest.fixture
def case():
    made = []

    def make(*a, **kw):
        made.append(Case(*a, **kw))
        return made[-1]
    yield make
    for c in made:
        c.e.close()


def test_records_that_cannot_be_allocated(case):
    rng = np.random.default_rng(3)
    c = case(_fact(rng.integers(0, 1 << 20, ROWS)), _query())
    c.e.fail_device_allocs(64 * MB, 1)     # the records take about 90 MB, the table 32
    assert c.run() == (0, 0)
    assert c.run() == (1, 0)


def test_records_come_back_after_an_overflow(case):
    """A quarter of the 1,024 partitions made for 1.8 million groups gets 4,700
    keys, more than their tables hold; the next execution knows of 3.7 million
    groups and makes twice as many partitions."""
    rng = np.random.default_rng(4)
    key = rng.integers(0, 2_100_000, ROWS) * 4_090
    key[0], key[1] = 1 << 33, 0
    c = case(_fact(key), _query())
    assert c.run() == (1, 0)
    keys = np.concatenate([(p << 23) + np.arange(4_700 if p % 4 == 0 else 3_255) * 1_700 for p in range(1024)])
    key = rng.permutation(np.concatenate([[1 << 33], keys, rng.choice(keys, ROWS - 1 - len(keys))]))
    c.change(key)
    assert c.run() == (1, 1)       # through the table in the end
    assert c.run() == (1, 0)
    assert c.run() == (1, 0)


def test_evenness_is_sampled_for_the_partitions_in_use(case):
    """Keys in every second range of 2^13: uneven over the partitions of that
    width that the first estimate asks for, even over the wider ones that the
    measured group count does."""
    rng = np.random.default_rng(5)
    pool = np.arange(1 << 24).reshape(-1, 1 << 13)[::2].ravel()
    key = rng.choice(rng.choice(pool, 300_000, replace=False), ROWS)
    key[0], key[1] = 0, (1 << 24) - 1
    c = case(_fact(key), _query())
    assert c.run() == (0, 0)
    assert c.run() == (1, 0)
    assert c.run() == (1, 0)


HLL_BYTES = 4 * 4096


def _first(c):
    s0 = c.e.stats()["d2h_bytes"]
    r = c.plan.execute()
    read = c.e.stats()["d2h_bytes"] - s0
    assert_matches_oracle(r, c.ref, c.q["aggs"])
    r.free()
    return read


@pytest.mark.parametrize("sel,counts", [(0.01, False), (0.2, True), (1.0, True)])
def test_distinct_keys_are_counted_where_the_rows_say_too_little(case, sel, counts):
    """Not under a selective filter, whose rows bound the groups better than a pass
    over every key is worth."""
    rng = np.random.default_rng(6)
    fact = _fact(rng.integers(0, 2_000_000, ROWS) * 1_000_003)
    fact["d"] = rng.integers(0, 1000, ROWS).astype(np.int32)
    c = case(fact, _query(dict(col="d", lo=0, hi=int(1000 * sel) - 1)))
    assert (_first(c) >= HLL_BYTES) == counts


def test_only_keys_that_pass_are_counted(case):
    """2 million keys, 20,000 of them in the rows that pass: the first execution's
    table is one for 20,000 groups."""
    rng = np.random.default_rng(7)
    d = rng.integers(0, 1000, ROWS).astype(np.int32)
    key = np.where(d < 200, rng.integers(0, 20_000, ROWS), rng.integers(0, 2_000_000, ROWS)) * 1_000_003
    fact = dict(_fact(key), d=d)
    c = case(fact, _query(dict(col="d", lo=0, hi=199)))
    assert _first(c) >= HLL_BYTES
    assert c.e.stats()["peak_reserved"] < 64 * MB
