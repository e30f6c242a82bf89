"""Grouping of the fan-out build: the key equal to a table's empty pattern, one
key holding every row, single-row runs, rows dropped by the predicate, several
batches of build rows; every table kind, against the oracle bit for bit."""
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


def _keys(rng, kind, n):
    if kind == "one":
        return np.full(n, 7)
    if kind == "unique":
        return rng.permutation(n) - n // 2
    if kind == "empty-pattern":
        return rng.integers(-3, 4, n)              # -1 is the empty pattern of both key widths
    return rng.integers(0, max(1, n // 3), n)


@pytest.mark.parametrize("kind", ["one", "unique", "empty-pattern", "mixed"])
@pytest.mark.parametrize("dt", [np.int32, np.int64])
@pytest.mark.parametrize("flags", [0, T.TP_FLAG_NO_DIRECT_JOIN, T.TP_FLAG_NO_STAGED | T.TP_FLAG_NO_DIRECT_JOIN])
@pytest.mark.parametrize("placement", [T.TP_DEVICE, T.TP_HOST_PAGES])
def test_runs_hold_every_admitted_row(kind, dt, flags, placement):
    rng = np.random.default_rng(5)
    n = 4_000
    m = 60 if kind in ("one", "empty-pattern") else 9_001   # run lengths stay moderate
    dim = dict(pk=_keys(rng, kind, m).astype(dt), attr=rng.integers(0, 25, m).astype(np.int32))
    fk = np.concatenate([rng.choice(dim["pk"], n - 500), rng.integers(-20_000, 20_000, 500).astype(dt)])
    fact = dict(fk=fk, v=rng.integers(0, 1000, n))
    q = dict(filter=None, join=dict(fact_col="fk", dim_col="pk", many=True), group=[("dim", "attr", 5)],
             dim_filter=dict(col="attr", lo=0, hi=19), aggs=[("sum", "v"), ("count",)])
    e = T.Engine(page_bytes=1 << 20, n_pages=64, flags=flags)
    try:
        ft = e.table_from_numpy(fact, placement=placement)
        d = e.table_from_numpy(dim, placement=placement, batch_rows=1_000)
        with e.plan(ft, d, q).execute() as r:
            assert_matches_oracle(r, oracle.run_query(fact, dim, q), q["aggs"])
    finally:
        e.close()
