"""Hints and estimates below the real number of groups: a key/value plan of
more than 2048 groups has a global table that takes some times more groups than
it was told of, whatever variant it chose."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2608_13696_gb300 import build as B
from paper_2608_13696_gb300 import rel


@pytest.fixture(scope="module")
def L():
    B.build()
    return rel.load()


def hint_plan(L, ops, key, hint, n_rows):
    cols = (rel.Col * 2)(rel.Col(0x1000, key, 0), rel.Col(0x2000, rel.I64, 0))
    keys = (ctypes.c_int32 * 1)(0)
    aggs = (rel.Agg * len(ops))(*[rel.Agg(rel.OPS[o], 1, 0, 0) for o in ops])
    d = rel.GroupByDesc(n_rows, 2, 1, 0, len(ops), cols, keys, (rel.RangePred * 1)(), aggs)
    p = rel.Plan()
    assert L.rel_plan_size(rel.OP_GROUPBY, ctypes.byref(d), 0, hint, None, 0, ctypes.byref(p),
                           None) == rel.REL_OK
    assert p.workspace_bytes == L.rel_plan_ws_bytes(ctypes.byref(p), len(ops), n_rows)
    return p


@pytest.mark.parametrize("ops", [("sum", "count"), ("sum", "count", "min", "max")])
@pytest.mark.parametrize("key", [rel.I64, rel.I32])
@pytest.mark.parametrize("hint", [2049, 3072, 3073, 5000, 5120, 5121, 20_000])
def test_global_slots(L, ops, key, hint):
    assert hint_plan(L, ops, key, hint, 10_000_000).slots >= 65536


@pytest.mark.parametrize("hint,bits", [(262_144, 8), (300_000, 8), (300_001, 9)])
def test_twice_the_groups_fit(L, hint, bits):
    p = hint_plan(L, ("sum", "count"), rel.I64, hint, 100_000_000)
    assert p.part_bits == bits
    assert p.slots >= 2 * hint - 1 or p.smem_slots >= 2 * (hint >> bits)


@pytest.mark.gpu
@pytest.mark.parametrize("ops", [("sum", "count"), ("sum", "count", "min", "max")])
@pytest.mark.parametrize("hint,groups", [(2049, 20_000), (5000, 20_000), (5120, 50_000), (9000, 50_000)])
@pytest.mark.parametrize("sketch", [0, rel.PLAN_SKETCH])
def test_answered(ops, hint, groups, sketch):
    from gpu_util import canon_groupby, query_to_cuda

    rng = np.random.default_rng(hint)
    n = 200_003  # sketched, the 9000 are one global table
    q = oracle.kv_query(rng.integers(0, groups, n) * 977, rng.integers(-100, 100, n), ops=ops)
    k, a = canon_groupby(*rel.groupby(query_to_cuda(q), groups_hint=hint, flags=sketch))
    ek, ea = oracle.groupby(q)
    np.testing.assert_array_equal(k, ek)
    np.testing.assert_array_equal(a, ea)
