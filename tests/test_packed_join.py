"""Packed 64-bit-key join tables: bucket overflow, missing keys, the key equal to
the empty pattern, payloads at the widest packed width and beyond it, errors,
and a predicate whose sample is wrong (the build finds the table too small and
the query runs again); every kernel path against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2508_05029_gb300 import theseus as T
from tests.helpers import assert_matches_oracle
from tests.test_jit_source import _compile, _nvrtc, _shape

FLAGS = [0, T.TP_FLAG_NO_JIT, T.TP_FLAG_NO_STAGED]


@pytest.mark.parametrize("shape", [_shape(join=4, ktype=1), _shape(join=4, ktype=0, lip=1),
                                   _shape(xjoins=((4, 1, 1), (4, 1, 0)), groups=((1, 0, 3), (1, 0, 4)), gdim=(1, 2, 0, 0)),
                                   _shape(sums=((0, 1, 0, 2, 0), (1, 1, 1, 3, 0), (1, 1, 1, 4, 0)))
                                   .replace("lo_only = false", "lo_only = false, wide = true")])
def test_nvrtc_compiles_packed_and_wide_shapes(shape):
    _compile(_nvrtc(), "#undef TP_ST_CONSUMERS\n#undef TP_ST_RPL\n#define TP_ST_CONSUMERS 31\n#define TP_ST_RPL 1\n" +
             shape + '#include "jit_dense.cuh"\n')


@pytest.fixture(scope="module")
def built():
    from paper_2508_05029_gb300 import build
    build.build()


def _tables(n, m, bits, seed=3):
    rng = np.random.default_rng(seed)
    pk = np.unique(rng.integers(-(1 << 62), 1 << 62, 2 * m))[:m]
    pk[: 2] = -1, 0
    rng.shuffle(pk)
    attr = rng.integers(0, 1 << bits, m)
    fk = rng.choice(pk, n)
    fk[:: 7] = rng.integers(-(1 << 62), 1 << 62, len(fk[:: 7]))
    return dict(fk=fk, v=rng.integers(0, 1000, n)), dict(pk=pk, attr=attr.astype(np.int32), sel=np.arange(m, dtype=np.int32))


def _query(bits, flt=None):
    return dict(filter=None, join=dict(fact_col="fk", dim_col="pk"), group=[("dim", "attr", bits)], dim_filter=flt,
                aggs=[("sum", "v"), ("count",)])


def _check(fact, dim, q, flags, retries=0, lf=0.0, **kw):
    e = T.Engine(page_bytes=4 << 20, n_pages=64, flags=flags)
    try:
        ft, dt = (e.table_from_numpy(t, placement=T.TP_DEVICE) for t in (fact, dim))
        p = e.plan(ft, dt, q, load_factor=lf, **kw)
        for _ in range(2):
            with p.execute() as r:
                assert_matches_oracle(r, oracle.run_query(fact, dim, q), q["aggs"])
        assert e.stats()["retries"] == retries
    finally:
        e.close()


@pytest.mark.gpu
@pytest.mark.parametrize("flags", FLAGS)
@pytest.mark.parametrize("m,bits,lf", [(2, 5, 0.0), (4096, 5, 0.0), (32_768, 5, 0.5), (32_769, 5, 0.5), (150_000, 8, 0.6),
                                       (150_000, 8, 0.9), (40_000, 12, 0.0), (40_000, 20, 0.0)])
def test_packed_join_matches_oracle(built, flags, m, bits, lf):
    fact, dim = _tables(60_001, m, bits)
    _check(fact, dim, _query(bits), flags, lf=lf)


@pytest.mark.gpu
@pytest.mark.parametrize("flags", FLAGS)
def test_a_sample_that_misses_the_admitted_rows(built, flags):
    """4096 evenly spaced rows see none of the admitted ones: the table is far
    too small, once, and the plan remembers it."""
    m = 4096 * 32
    fact, dim = _tables(60_001, m, 5)
    dim["sel"] = (np.arange(m) % 32 != 0).astype(np.int32)
    _check(fact, dim, _query(5, flt=dict(col="sel", lo=1, hi=1)), flags, retries=1)


@pytest.mark.gpu
@pytest.mark.parametrize("flags", FLAGS)
def test_errors_of_a_packed_join(built, flags):
    fact, dim = _tables(20_001, 30_000, 5)
    e = T.Engine(flags=flags, page_bytes=4 << 20, n_pages=64)
    try:
        ft = e.table_from_numpy(fact, placement=T.TP_DEVICE)
        bad = dict(dim, attr=np.full(30_000, 32, np.int32))     # does not fit 5 bits
        with pytest.raises(T.TPError) as err:
            e.plan(ft, e.table_from_numpy(bad, placement=T.TP_DEVICE), _query(5)).execute()
        assert err.value.code == T.TP_E_RANGE
        twice = dict(dim, pk=np.where(np.arange(30_000) == 17, dim["pk"][29_000], dim["pk"]))
        with pytest.raises(T.TPError) as err:
            e.plan(ft, e.table_from_numpy(twice, placement=T.TP_DEVICE), _query(5)).execute()
        assert err.value.code == T.TP_E_DUP_KEY
    finally:
        e.close()


@pytest.mark.parametrize("selected", ["", "#define TPJ_SELECTED 1\n"])
@pytest.mark.parametrize("shape", [
    _shape(groups=((0, 1, 64),), sums=((1, 1, 1, 0, 0),), fast=False),
    _shape(join=4, ktype=1, groups=((0, 0, 10), (0, 1, 10)), fast=False,
           sums=((0, 1, 0, 0, 0), (0, 2, 0, 0, 0), (1, 1, 0, 0, 0), (0, 0, 0, 0, 0))),
    _shape(join=0, filter=0, groups=((0, 1, 64),), sums=(), fast=False)])
def test_nvrtc_compiles_record_scans(shape, selected, monkeypatch):
    from tests import test_jit_source
    monkeypatch.setattr(test_jit_source, "HEADERS", test_jit_source.HEADERS + ["records.cuh", "jit_records.cuh"])
    _compile(_nvrtc(), "#undef TP_ST_CONSUMERS\n#undef TP_ST_RPL\n#define TP_ST_CONSUMERS 8\n#define TP_ST_RPL 4\n" +
             selected + shape + '#include "jit_records.cuh"\n')
