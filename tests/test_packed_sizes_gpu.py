"""Packed join tables sized by a dimension predicate's pass rate: over a whole
octave of rates the reservation stays one for the admitted rows."""
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


@pytest.mark.parametrize("percent", [11.0, 13.0, 14.0, 14.3, 14.6, 15.0, 16.0, 20.0, 22.0])
def test_reservation_follows_the_admitted_rows(percent):
    rng = np.random.default_rng(int(percent * 10))
    n, m = 20_001, 2_000_000
    dim = dict(pk=rng.permutation(m) * 0x9E3779B97B, attr=rng.integers(0, 25, m).astype(np.int32),
               d=rng.integers(0, 1000, m).astype(np.int32))
    fact = dict(fk=rng.choice(dim["pk"], n), v=rng.integers(0, 1000, n))
    q = dict(filter=None, join=dict(fact_col="fk", dim_col="pk"), group=[("dim", "attr", 5)],
             dim_filter=dict(col="d", lo=0, hi=int(percent * 10) - 1), aggs=[("sum", "v"), ("count",)])
    import torch
    e = T.Engine()
    try:
        ft, dt = (e.table_from_torch({k: torch.from_numpy(v).cuda() for k, v in t.items()}) for t in (fact, dim))
        torch.cuda.synchronize()
        with e.plan(ft, dt, q, lip=T.TP_LIP_OFF).execute() as r:
            assert_matches_oracle(r, oracle.run_query(fact, dim, q), q["aggs"])
        # half a million words or a million, where all rows unpacked take 64 MB
        assert e.stats()["peak_reserved"] < 8 * 2 * MB + 1 * MB
        assert e.stats()["retries"] == 0
    finally:
        e.close()
