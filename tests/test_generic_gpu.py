"""GPU parity of the descriptor-driven group-by and its distinct count: every
column type in every role, filters whose bounds lie outside the column's type,
groups that fit the CTA's table, that overfill it and that exceed it, one- and
two-byte keys (the bit-per-key count), rows around the chunk edges, unaligned
columns.  Exact int64: the tolerance is zero."""
import numpy as np
import pytest

import oracle
from paper_2608_13696_gb300 import rel

from gpu_util import canon_groupby, cuda, query_to_cuda

pytestmark = pytest.mark.gpu
I64 = np.iinfo(np.int64)


def make(n, seed, groups):
    rng = np.random.default_rng(seed)
    wide = rng.integers(I64.min, I64.max, n)
    return [rng.integers(0, 7, n).astype(np.uint8), rng.integers(0, 256, n).astype(np.uint8),
            rng.integers(-groups // 2, groups // 2 + 1, n).astype(np.int32),
            rng.integers(-(2**31), 2**31, n).astype(np.int32),
            rng.integers(-groups, groups, n) * 2**33, wide]


AGGS = [("sum", 5, [(3, 7, -3)]), ("min", 3, []), ("max", 5, [(1, 1, 1), (2, 0, 2)]), ("count", 0, []),
        ("sum", 1, [])]
QUERIES = {
    "u8": ([1], [(3, -(2**40), 2**40)], AGGS[:2]),
    "u8u8": ([0, 1], [(2, -50, 2**35)], AGGS),
    "u8u8_none_pass": ([0, 1], [(3, 2**33, 2**34)], AGGS[:3]),
    "u8i32": ([0, 2], [(1, 10, 250), (5, I64.min + 1, I64.max)], AGGS),
    "i32u8u8": ([2, 1, 0], [], AGGS[2:4]),
    "i64": ([4], [(1, -5, 300), (3, -(2**31), 2**30), (0, 1, 6)], AGGS + AGGS[:3]),
    "i32_minmax": ([2], [], [("min", 5, []), ("max", 5, [])]),
}


@pytest.mark.parametrize("name", list(QUERIES))
@pytest.mark.parametrize("n,groups", [(1, 1), (511, 3), (4099, 40), (50_003, 4000), (120_001, 60_000)])
@pytest.mark.parametrize("offset", [0, 1])
def test_matches_oracle(name, n, groups, offset):
    keys, preds, aggs = QUERIES[name]
    cols = make(n + offset, n + len(name), groups)
    q = {"cols": [c[offset:] for c in cols], "keys": keys, "preds": preds, "aggs": aggs}
    ek, ea = oracle.groupby(q)
    qc = dict(q)
    qc["cols"] = [cuda(c)[offset:] for c in cols]  # offset 1: off 16-byte alignment
    for flags in (rel.PLAN_EXACT, 0, rel.PLAN_GENERIC | rel.PLAN_EXACT):
        p = rel.plan_groupby(qc, flags=flags)
        if flags & rel.PLAN_EXACT:
            assert p.est_groups == len(ek)
        if p.smem_slots:
            p.smem_slots = max(16, p.smem_slots)  # the smallest table a plan may name
        gk, ga = canon_groupby(*rel.groupby(qc, plan=p))
        np.testing.assert_array_equal(gk, ek)
        np.testing.assert_array_equal(ga, ea)


@pytest.mark.parametrize("smem,variant", [(0, rel.VAR_GLOBAL), (2048, rel.VAR_GLOBAL), (16, rel.VAR_SMEM)])
def test_layers_and_overflow(smem, variant):
    q = {"cols": make(30_000, 5, 9000), "keys": [0, 2], "preds": [], "aggs": AGGS}
    ek, ea = oracle.groupby(q)
    qc = query_to_cuda(q)
    p = rel.plan_groupby(qc, groups_hint=len(ek)).layers(0, smem, variant)
    gk, ga = canon_groupby(*rel.groupby(qc, plan=p))
    np.testing.assert_array_equal(gk, ek)
    np.testing.assert_array_equal(ga, ea)
    p.slots = 4096  # fewer than the groups
    with pytest.raises(rel.RelError) as e:
        rel.groupby(qc, plan=p)
    assert e.value.status == rel.REL_E_OVERFLOW


@pytest.mark.parametrize("n", [1, 3, 1023, 3073, 700_001])
@pytest.mark.parametrize("pins", [1, 3, 6])
@pytest.mark.parametrize("offset", [0, 1])
def test_fused_shape_with_pinned_groups(n, pins, offset):
    """All groups pinned, some pinned (the others take the global table), rows
    around the chunk edges, unaligned columns, extreme values."""
    import synth
    from paper_2608_13696_gb300 import workloads

    li = synth.lineitem(n + offset, seed=n + pins)
    li["price"][:: 97] = I64.max
    li["qty"][1:: 89] = I64.min
    q = oracle.lineitem_query({k: v[offset:] for k, v in li.items()})
    ek, ea = oracle.groupby(q)
    qc = workloads.lineitem_query({k: cuda(v)[offset:] for k, v in li.items()})
    p = rel.plan_groupby(qc, groups_hint=6).layers(8, 0, rel.VAR_SMEM)
    keys = [0, 1, 256, 257, 512, 513][:pins]
    for mult in range(0x9E3779B1, 0x9E3779B1 + 2 * 4096, 2):  # a multiplier without collisions
        f = [((((k ^ (1 << 31)) & 0xFFFFFFFF) * (mult & 0xFFFFFFFF)) >> 32) & 7 for k in keys]
        if len(set(f)) == len(f):
            break
    p.tiny_mult = mult & 0xFFFFFFFF
    p.n_hot = len(keys)
    for i, k in enumerate(keys):
        p.hot_keys[i] = k
    gk, ga = canon_groupby(*rel.groupby(qc, plan=p))
    np.testing.assert_array_equal(gk, ek)
    np.testing.assert_array_equal(ga, ea)
