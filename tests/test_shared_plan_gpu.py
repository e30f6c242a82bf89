"""One plan run by a server's lane and by tp_execute at the same time, from its
first execution on: every result against the oracle bit for bit."""
import threading

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


@pytest.mark.parametrize("placement", [T.TP_DEVICE, T.TP_HOST_PAGES])
def test_a_plan_on_two_lanes(placement):
    rng = np.random.default_rng(8)
    n, m = 40_001, 3_000
    fact = dict(fk=rng.integers(0, m, n), v=rng.integers(0, 1000, n), d=rng.integers(0, 100, n).astype(np.int32))
    dim = dict(pk=np.arange(m) * 1, attr=rng.integers(0, 25, m).astype(np.int32))
    e = T.Engine(page_bytes=1 << 20, n_pages=64, batch_rows=9_001)
    try:
        ft, dt = (e.table_from_numpy(t, placement=placement) for t in (fact, dim))
        srv = T.Server(e, workers=2, cache_dims=False)
        for k in range(20):
            q = dict(filter=dict(col="d", lo=0, hi=50 + k), join=dict(fact_col="fk", dim_col="pk"),
                     group=[("dim", "attr", 5 + k % 3)], aggs=[("sum", "v"), ("count",)])
            p = e.plan(ft, dt, q)
            ref = oracle.run_query(fact, dim, q)
            failed = []

            def here():
                try:
                    for _ in range(3):
                        with p.execute() as r:
                            assert_matches_oracle(r, ref, q["aggs"])
                except Exception as x:   # noqa: BLE001 -- reported below
                    failed.append(x)

            th = threading.Thread(target=here)
            tickets = [srv.submit(p) for _ in range(3)]
            th.start()
            for t in tickets:
                r, _ = srv.wait(t)
                assert_matches_oracle(r, ref, q["aggs"])
                r.free()
            th.join()
            assert not failed, failed
        srv.stop()
    finally:
        e.close()
