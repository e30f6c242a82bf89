"""Sums that may leave int64 as 32-bit limbs in the run-time compiled dense
kernel: terms at the edges of three limbs (span just below and at 2^64, with
and without an offset that fits int64) and of four, one and several rows per
group, against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2508_05029_gb300 import theseus as T
from tests.helpers import assert_matches_oracle

pytestmark = pytest.mark.gpu

I64 = (-(1 << 63), (1 << 63) - 1)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_05029_gb300 import build
    build.build()


def _col(rng, n, lo, hi):
    x = rng.integers(lo, hi, n, dtype=np.int64, endpoint=True)
    x[0], x[-1] = lo, hi
    return x


@pytest.mark.parametrize("a,b,k", [
    (I64, (0, 0), 1),                             # plain sum of the whole int64 range: span 2^64 - 1
    (I64, (0, 1), 1),                             # product: span beyond 2^64, four limbs
    ((0, (1 << 62)), (-2, 1), 1),                 # products up to 3 * 2^62: three limbs
    ((-(1 << 62), 1 << 62), (-(1 << 62), 1 << 62), -7),
    ((1 << 61, 1 << 62), I64, 1 << 62),           # |k - b| beyond int64
    ((5, 900), (0, 10), 100),                     # narrow next to the wide one
])
@pytest.mark.parametrize("n,many_groups", [(1536, False), (4 * 152 * 1536 + 777, True)])
def test_limb_sums_match_oracle(a, b, k, n, many_groups):
    rng = np.random.default_rng(n + k % 1000)
    fact = dict(a=_col(rng, n, *a), b=_col(rng, n, *b), w=_col(rng, n, *I64), q=_col(rng, n, 0, 5000),
                f=(rng.integers(0, 200, n) if many_groups else np.zeros(n)).astype(np.uint8))
    q = dict(filter=None, join=None, group=[("fact", "f", 8)],
             aggs=[("sum_mul_sub", "a", k, "b"), ("sum", "w"), ("avg", "q"), ("count",), ("avg", "w")])
    e = T.Engine()
    try:
        t = _device(e, fact)
        p = e.plan(t, None, q)
        with p.execute() as r:
            assert_matches_oracle(r, oracle.run_query(fact, None, q), q["aggs"])
        assert e.stats()["jit_launches"] == 1
    finally:
        e.close()


def _device(e, cols):
    import torch
    return e.table_from_torch({k: torch.from_numpy(v).cuda() for k, v in cols.items()})
