"""A request that comes alone when the budget is taken up by join tables the
server keeps from earlier batches: they make room for it."""
import numpy as np
import pytest

import oracle
from paper_2508_05029_gb300 import theseus as T
from tests.helpers import assert_matches_oracle

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_05029_gb300 import build
    build.build()


@pytest.mark.parametrize("fact_rows", [50_001, 4 * MB + 3])   # the dispatcher's own lane; a worker's lane
def test_idle_join_tables_make_room(fact_rows):
    rng = np.random.default_rng(9)
    e = T.Engine(page_bytes=1 * MB, n_pages=64)
    cases = []
    for k, n in enumerate([50_001] * 4 + [fact_rows]):
        m = 500_000
        dim = dict(pk=rng.permutation(m) * 0x9E3779B97B + k, attr=rng.integers(0, 25, m).astype(np.int32))
        fact = dict(fk=rng.choice(dim["pk"], n), v=rng.integers(0, 1000, n))
        q = dict(filter=None, join=dict(fact_col="fk", dim_col="pk"), group=[("dim", "attr", 5)],
                 aggs=[("sum", "v"), ("count",)])
        ft, dt = (e.table_from_numpy(t, placement=T.TP_DEVICE) for t in (fact, dim))
        cases.append((e.plan(ft, dt, q), oracle.run_query(fact, dim, q), q, ft, dt))
    used, cap = e.budget()
    srv = T.Server(e, workers=1, cache_dims=False, batch=True)

    def check(ticket, case):
        r, _ = srv.wait(ticket, timeout_s=60)
        with r:
            assert_matches_oracle(r, case[1], case[2]["aggs"])
    try:
        for _ in range(20):
            for t, c in [(srv.submit(c[0]), c) for c in cases[:4] * 4]:
                check(t, c)
            if srv.stats()["batches"] > 0 and e.budget()[0] - used >= 16 * MB:
                break
        kept = e.budget()[0]
        assert kept - used >= 16 * MB        # at least one table of a million 16-byte slots
        e.set_budget(kept + 4 * MB)          # the next request needs 8 MB
        check(srv.submit(cases[4][0]), cases[4])
        assert srv.stats()["failed"] == 0
    finally:
        srv.stop()
        e.close()
