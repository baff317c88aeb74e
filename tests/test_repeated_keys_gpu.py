"""Inputs in which neighbouring rows have one key: warps that combine their rows
before the shared-memory adds (shared table, partition aggregation, the
descriptor-driven kernel), and plans whose pinned keys are all the keys of the
sample, with rows of other keys beside them.  Values are any int64, so sums
wrap and minima and maxima are extreme.  Exact: the tolerance is zero."""
import numpy as np
import pytest

import oracle
from paper_2608_13696_gb300 import rel

from gpu_util import canon_groupby, cuda

pytestmark = pytest.mark.gpu
I64 = np.iinfo(np.int64)
OPS = {1: ("min",), 2: ("sum", "count"), 3: ("sum", "max", "sum"), 4: ("max", "sum", "min", "count")}


def ranks(kind, n, groups, rng):
    if kind == "one":
        return np.zeros(n, np.int64)
    if kind == "one_but":  # few rows of other keys, in the first and later chunks
        r = np.zeros(n, np.int64)
        r[rng.random(n) < 0.002] = 1
        return r
    length = {"runs64": 64, "runs37": 37, "runs128": 128}[kind]
    return np.repeat(rng.integers(0, groups, n // length + 1), length)[:n]


def check(k, v, ops, offset=0, **kw):
    q = {"cols": [cuda(k)[offset:], cuda(v)[offset:]], "keys": [0], "preds": [],
         "aggs": [(o, 1, []) for o in ops]}
    p = rel.plan_groupby(q, **kw)
    gk, ga = canon_groupby(*rel.groupby(q, plan=p))
    ek, ea = oracle.groupby(oracle.kv_query(k[offset:], v[offset:], ops=ops))
    np.testing.assert_array_equal(gk, ek)
    np.testing.assert_array_equal(ga, ea)
    return p


@pytest.mark.parametrize("na", [1, 2, 3, 4])
@pytest.mark.parametrize("dtype", [np.int64, np.int32])
@pytest.mark.parametrize("kind", ["one", "one_but", "runs64", "runs37", "runs128"])
@pytest.mark.parametrize("n", [63, 4096, 250_001, 1_300_000])
def test_shared_table(na, dtype, kind, n):
    rng = np.random.default_rng(n + na)
    k = (ranks(kind, n, 5, rng) * 7919 - 3).astype(dtype)
    v = rng.integers(I64.min, I64.max, n, endpoint=True)
    for offset in (0, 1):
        check(k, v, OPS[na], offset, groups_hint=5)


@pytest.mark.parametrize("na", [2, 4])
@pytest.mark.parametrize("kind", ["runs64", "runs37"])
@pytest.mark.parametrize("n,groups,bits", [(300_007, 3000, 4), (1_000_003, 20_000, 10)])
def test_partitioned(na, kind, n, groups, bits):
    rng = np.random.default_rng(n + na)
    k = ranks(kind, n, groups, rng) * 7919 - 3
    k[::1000] = I64.min
    v = rng.integers(I64.min, I64.max, n, endpoint=True)
    p = check(k, v, OPS[na], groups_hint=3100 if bits == 4 else 500_000,
              flags=rel.plan_force(rel.VAR_PARTITIONED))
    assert p.part_bits == bits


@pytest.mark.parametrize("na", [2, 4])
@pytest.mark.parametrize("dtype", [np.int64, np.int32])
@pytest.mark.parametrize("n", [5000, 100_003, 900_001])
@pytest.mark.parametrize("keys", [1, 3, 8])
@pytest.mark.parametrize("hint", [25, 500])
def test_every_sampled_key_pinned(na, dtype, n, keys, hint):
    rng = np.random.default_rng(n + keys)
    k = rng.integers(0, keys, n).astype(dtype) * 31
    # other keys between the sample's windows of 64 rows: few, and more than the table holds
    free = np.ones(n, bool)
    for w in range(64):
        s = w * (n - 64) // 63
        free[s:s + 64] = False
    rows = np.flatnonzero(free)[::3]
    k[rows] = 1000 + rng.integers(0, {25: 20, 500: 1500}[hint], len(rows)).astype(dtype)
    if dtype == np.int64:
        k[rows[::7]] = I64.min
    v = rng.integers(I64.min, I64.max, n, endpoint=True)
    q = {"cols": [cuda(k), cuda(v)], "keys": [0], "preds": [], "aggs": [(o, 1, []) for o in OPS[na]]}
    p = rel.plan_groupby(q, groups_hint=hint, flags=rel.PLAN_SKETCH)
    assert p.flags & rel.PLAN_SAMPLE_PINNED and p.n_hot == keys and p.smem_slots > 0
    p.slots = 4096
    p.workspace_bytes = 0  # of the larger table, asked for again
    gk, ga = canon_groupby(*rel.groupby(q, plan=p))
    ek, ea = oracle.groupby(oracle.kv_query(k, v, ops=OPS[na]))
    np.testing.assert_array_equal(gk, ek)
    np.testing.assert_array_equal(ga, ea)
