"""Device memory a lane keeps between executions: it stays inside the device
budget beside the reservations, makes room for whatever else is allocated, and
is as large as the most an execution held at once.  Memory in use is read from
the device's memory pool."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2508_05029_gb300 import theseus as T
from tests.helpers import assert_matches_oracle

pytestmark = pytest.mark.gpu
MB = 1 << 20
USED_CURRENT, USED_HIGH = 7, 8   # CUmemPool_attribute


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_05029_gb300 import build
    build.build()


class Pool:
    def __init__(self):
        import torch
        torch.zeros(1, device="cuda")
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.h = ctypes.c_void_p()
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.h), 0) == 0

    def get(self, attr=USED_CURRENT):
        v = ctypes.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.h, attr, ctypes.byref(v)) == 0
        return v.value

    def reset_high(self):
        v = ctypes.c_uint64(0)
        assert self.cu.cuMemPoolSetAttribute(self.h, USED_HIGH, ctypes.byref(v)) == 0


def _wrap(e, cols):
    import torch
    dev = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in cols.items()}
    t = e.table_from_torch(dev)
    torch.cuda.synchronize()
    return t


def _star(e, m, n=20_001):
    """A join to m rows of sparse 64-bit keys (a packed table of 8 bytes per slot)."""
    rng = np.random.default_rng(m)
    dim = dict(pk=rng.permutation(m).astype(np.int64) * 0x9E3779B97B, attr=rng.integers(0, 25, m).astype(np.int32))
    fact = dict(fk=rng.choice(dim["pk"], n), v=rng.integers(0, 1000, n))
    q = dict(filter=None, join=dict(fact_col="fk", dim_col="pk"), group=[("dim", "attr", 5)],
             aggs=[("sum", "v"), ("count",)])
    ft, dt = _wrap(e, fact), _wrap(e, dim)
    p = e.plan(ft, dt, q, join_partitions=1)
    ref = oracle.run_query(fact, dim, q)

    def run():
        assert ft.h and dt.h      # the tables own the tensors
        with p.execute() as r:
            assert_matches_oracle(r, ref, q["aggs"])
    return run


def _engine(budget=0, **kw):
    return T.Engine(page_bytes=4 * MB, n_pages=64, device_budget_bytes=budget, **kw)


def test_a_smaller_budget_takes_the_arena_back():
    pool, e = Pool(), _engine()
    try:
        base = pool.get()
        run = _star(e, 3_000_000)
        run()
        run()
        assert pool.get() - base >= 64 * MB       # kept between executions
        e.set_budget(100 * MB)
        assert pool.get() - base <= 12.5 * MB     # an eighth of the budget at most
        run()
        assert pool.get() - base <= 12.5 * MB
    finally:
        e.close()


def test_reservations_and_arena_stay_inside_the_budget():
    pool, e = Pool(), _engine(67 * MB)
    try:
        small, large = _star(e, 140_000), _star(e, 3_000_000)   # tables of 4 and 64 MB
        base = pool.get()
        small()
        small()
        assert pool.get() - base >= 4 * MB
        pool.reset_high()
        large()
        assert pool.get(USED_HIGH) - base <= 67 * MB
        small()
        t = e.table_from_numpy(dict(a=np.arange(8 * MB)), placement=T.TP_DEVICE)    # 64 MB reserved
        assert pool.get() - base <= 67 * MB    # once placed: widening its pages takes a buffer beside the reservation
        t.destroy()
    finally:
        e.close()


def test_a_failed_allocation_runs_without_the_arena():
    e = _engine()
    try:
        small, large = _star(e, 140_000), _star(e, 3_000_000)
        small()
        e.fail_device_allocs(32 * MB, 1)
        large()
        assert e.stats()["retries"] == 1
        huge = _star(e, 6_000_000)
        e.fail_device_allocs(64 * MB, 2)   # without the arena too
        with pytest.raises(T.TPError) as err:
            huge()
        assert err.value.code == T.TP_E_CUDA
        huge()
    finally:
        e.close()


def test_an_idle_lane_gives_its_arena_to_another_allocation():
    pool, e = Pool(), _engine()
    try:
        rng = np.random.default_rng(1)
        _star(e, 3_000_000)()
        held = pool.get()
        e.fail_device_allocs(8 * MB, 1)
        a = rng.integers(0, 100, 2 * MB)
        t = e.table_from_numpy(dict(a=a), placement=T.TP_DEVICE)     # 16 MB: fails once, then has the arena's room
        assert pool.get() <= held - 48 * MB
        t.destroy()
    finally:
        e.close()


def test_the_arena_is_as_large_as_the_peak():
    """A group table that overflows three times: the tables dropped on the way
    are not part of what the next execution needs."""
    pool = Pool()
    rng = np.random.default_rng(2)
    n, groups = 600_000, 300_000
    fact = dict(k=rng.integers(0, groups, n), v=rng.integers(0, 1000, n))
    q = dict(filter=None, join=None, group=[("fact", "k", 40)], aggs=[("sum", "v")])
    ref = oracle.run_query(fact, None, q)
    peak = None
    for budget in (100 * MB, 0):     # the first leaves no room for an arena
        e = _engine(budget, flags=T.TP_FLAG_NO_DIRECT_AGG)
        try:
            t = _wrap(e, fact)
            p = e.plan(t, None, q, expected_groups=1_000)
            base = pool.get()
            pool.reset_high()
            with p.execute() as r:
                assert_matches_oracle(r, ref, q["aggs"])
            assert e.stats()["retries"] == 3
            if peak is None:
                assert pool.get() == base
                peak = pool.get(USED_HIGH) - base - ref.n_groups * 32    # beside the result
            else:
                assert 0 < pool.get() - base <= peak + 2 * MB
            for _ in range(2):
                with p.execute() as r:
                    assert_matches_oracle(r, ref, q["aggs"])
        finally:
            e.close()
