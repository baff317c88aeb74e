"""GPU parity of the shared-memory aggregate table and the kernels around it:
the streaming group-by with a CTA-shared table, the partition aggregation
(equal pieces of the records, further pieces of oversized partitions) and the
batched group-by and join.  All results are exact int64, so the tolerance is
zero.  Sizes sit at the edges: one row, partial chunks, tables that are just
full and just too small, one key in every row, extreme values."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_13696_gb300 import rel

from gpu_util import canon_groupby, canon_join, cuda, query_to_cuda

pytestmark = pytest.mark.gpu
OPS = {2: ("sum", "count"), 4: ("max", "sum", "min", "count")}
I64 = np.iinfo(np.int64)


def column(kind, n, groups, dtype, seed):
    rng = np.random.default_rng(seed)
    if kind == "skewed":  # half the rows on one key
        r = np.where(rng.random(n) < 0.5, 1, rng.integers(0, groups, n))
    else:
        r = rng.integers(0, groups, n)
    k = (r.astype(np.int64) * np.int64(0x9E3779B97F4A7C15 - 2**64)) if dtype == np.int64 \
        else (r * 7919 - 1000).astype(np.int32)
    if dtype == np.int64 and n > 2:
        k[:: max(3, n // 5)] = I64.min
    v = rng.integers(-(2**20), 2**20, n)
    v[rng.random(n) < 0.05] = I64.min  # sums wrap, both halves of the word carry
    v[rng.random(n) < 0.05] = I64.max
    return k, v


def check(q, plan=None, **kw):
    qc = query_to_cuda(q)
    if plan is None:
        plan = rel.plan_groupby(qc, **kw)
    k, a = canon_groupby(*rel.groupby(qc, plan=plan))
    ek, ea = oracle.groupby(q)
    np.testing.assert_array_equal(k, ek)
    np.testing.assert_array_equal(a, ea)
    return plan


@pytest.mark.parametrize("na", [2, 4])
@pytest.mark.parametrize("dtype", [np.int64, np.int32])
@pytest.mark.parametrize("n,groups,slots", [(1, 1, 16), (1023, 16, 16), (40_961, 300, 256),
                                            (70_003, 2048, 4096), (50_000, 9000, 4096)])
def test_stream_shared_table(na, dtype, n, groups, slots):
    k, v = column("uniform", n, groups, dtype, n + na)
    q = oracle.kv_query(k, v, ops=OPS[na])
    p = rel.plan_groupby(query_to_cuda(q), groups_hint=max(groups, 1))
    check(q, plan=p.layers(8, slots, rel.VAR_SMEM))


@pytest.mark.parametrize("na", [2, 4])
def test_stream_shared_table_grows_on_large_inputs(na):
    """Enough rows for the wider table, the columns off 16-byte alignment."""
    n = 2_600_011
    k, v = column("skewed", n, 700, np.int64, 3)
    for off in (0, 1):
        q = {"cols": [cuda(k)[off:], cuda(v)[off:]], "keys": [0], "preds": [],
             "aggs": [(o, 1, []) for o in OPS[na]]}
        got = canon_groupby(*rel.groupby(q, groups_hint=701, flags=rel.PLAN_SKETCH))
        exp = oracle.groupby(oracle.kv_query(k[off:], v[off:], ops=OPS[na]))
        np.testing.assert_array_equal(got[0], exp[0])
        np.testing.assert_array_equal(got[1], exp[1])


@pytest.mark.parametrize("na", [2, 4])
@pytest.mark.parametrize("kind", ["uniform", "skewed"])
@pytest.mark.parametrize("n,groups,hint", [(100, 60, 5000), (30_007, 5000, 5000),
                                           (200_003, 60_000, 60_000), (200_003, 9000, 5000),
                                           (400_001, 150_000, 300_000)])
def test_partitioned_pieces(na, kind, n, groups, hint):
    """Equal pieces (few partitions), whole partitions and the pieces of an
    oversized one, with tables that hold the keys and that do not."""
    k, v = column(kind, n, groups, np.int64, groups)
    q = oracle.kv_query(k, v, ops=OPS[na])
    check(q, groups_hint=hint, flags=rel.plan_force(rel.VAR_PARTITIONED))


@pytest.mark.parametrize("na", [2, 4])
def test_partitioned_plan_with_a_small_spill_table(na):
    """A plan whose global table cannot take every piece keeps whole partitions."""
    k, v = column("skewed", 50_021, 3000, np.int64, 8)
    q = oracle.kv_query(k, v, ops=OPS[na])
    p = rel.plan_groupby(query_to_cuda(q), groups_hint=3100,
                         flags=rel.plan_force(rel.VAR_PARTITIONED))
    p.slots = 2048
    check(q, plan=p)


@pytest.mark.parametrize("cfg", [(128, 4, 1, 512), (512, 8, 1, 2048), (256, 4, 4, 512), (512, 16, 1, 0)])
@pytest.mark.parametrize("ops", [["sum", "count"], ["min", "sum"], ["max", "min", "count", "sum"],
                                 ["count"]])
def test_batch_group_by_edges(cfg, ops):
    cols = [column(kind, n, g, dt, n) for kind, n, g, dt in
            (("uniform", 1, 1, np.int64), ("skewed", 5003, 40, np.int32),
             ("uniform", 70_001, 500, np.int64), ("uniform", 30_000, 1500, np.int32),
             ("skewed", 66_000, 30_000, np.int64), ("uniform", 2047, 2047, np.int64))]
    gs = []
    for k, v in cols:
        g = len(np.unique(k))
        gs.append({"keys": cuda(k), "vals": None if ops == ["count"] else cuda(v), "ops": ops,
                   "slots": 1 << max(4, (2 * g - 1).bit_length()), "est_groups": g,
                   "capacity": g + 1})
    b = rel.Batch(gs, []).prepare(cfg)
    b.run()
    counts, flags = b.results()
    assert not any(flags)
    for i, (k, v) in enumerate(cols):
        gk, ga = canon_groupby(*b.groupby_output(i, counts[i]))
        ek, ea = oracle.groupby(oracle.kv_query(k, v, ops=ops))
        np.testing.assert_array_equal(gk, ek)
        np.testing.assert_array_equal(ga, ea)


@pytest.mark.parametrize("items", [4, 16])
def test_batch_join_edges(items):
    """Unique and repeated build keys, sectors that fill up, INT64_MIN on both
    sides, one-row sides."""
    rng = np.random.default_rng(items)
    sides = []
    for nb, npr, dom in ((1, 1, 1), (1000, 4099, 1000), (5000, 9001, 60), (40_000, 70_003, 200_000)):
        bk = rng.integers(0, dom, nb) * 977 - 5
        pk = rng.integers(0, dom + 3, npr) * 977 - 5
        bk[:: max(2, nb // 3)] = I64.min
        pk[:: max(2, npr // 4)] = I64.min
        sides.append((bk, rng.integers(0, I64.max, nb), pk))
    exp = [oracle.join(*s) for s in sides]
    b = rel.Batch([], [{"build_keys": cuda(a), "build_payload": cuda(p), "probe_keys": cuda(c),
                        "capacity": len(e[0]) + 1} for (a, p, c), e in zip(sides, exp)],
                  device="cuda").prepare((256, items, 1, 512))
    b.run()
    counts, flags = b.results()
    assert not any(flags)
    for i, e in enumerate(exp):
        got = canon_join(*b.join_output(i, counts[i]))
        for x, y in zip(got, e):
            np.testing.assert_array_equal(x, y)
    torch.cuda.synchronize()


@pytest.mark.parametrize("na", [2, 4])
@pytest.mark.parametrize("dtype", [np.int64, np.int32])
@pytest.mark.parametrize("n", [5, 511, 3073, 700_003])
@pytest.mark.parametrize("groups", [1, 4, 6])
def test_all_groups_pinned(na, dtype, n, groups):
    """The pinned kernel, with rows the sample missed and INT64_MIN / INT64_MAX keys."""
    k, v = column("uniform", n, groups, dtype, n + groups)
    if dtype == np.int64:
        k[n // 2] = I64.max
    k[n - 1] = 12345  # one row of one more key
    for off in (0, 1):
        q = oracle.kv_query(k[off:], v[off:], ops=OPS[na])
        qc = {"cols": [cuda(k)[off:], cuda(v)[off:]], "keys": [0], "preds": [],
              "aggs": [(o, 1, []) for o in OPS[na]]}
        p = rel.plan_groupby(qc, groups_hint=max(4, groups), flags=rel.PLAN_SKETCH)
        got = canon_groupby(*rel.groupby(qc, plan=p, capacity=64))
        exp = oracle.groupby(q)
        np.testing.assert_array_equal(got[0], exp[0])
        np.testing.assert_array_equal(got[1], exp[1])


@pytest.mark.parametrize("n", [33, 4096, 4097, 60_001])
@pytest.mark.parametrize("groups", [1, 200, 50_000])
@pytest.mark.parametrize("dtype", [np.int64, np.int32])
def test_exact_plan_with_sketch(n, groups, dtype):
    """The exact count beside the sketch, and in its place on small inputs."""
    k, v = column("uniform", n, groups, dtype, n)
    s = oracle.sketch(oracle.kv_query(k, v))
    for keys in ([0], [0, 2]):
        if len(keys) == 2 and dtype == np.int64:
            continue
        cols = [cuda(k), cuda(v), cuda((k % 7).astype(np.uint8))]
        q = {"cols": cols, "keys": keys, "preds": [], "aggs": [("sum", 1, []), ("count", 1, [])]}
        p = rel.plan_groupby(q, flags=rel.PLAN_EXACT | rel.PLAN_SKETCH)
        assert p.est_groups == len(np.unique(k))  # the second column follows from the first
        if len(keys) == 1:
            assert set(p.hot_keys[i] for i in range(p.n_hot)) <= set(int(x) for x in s["top_key"])
