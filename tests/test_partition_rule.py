"""When the partition aggregation works on equal pieces of the records (which
meet in the global table) and when on whole partitions: by the rows a partition
has.  Plans need no GPU; results on both sides of the line do, and are exact
int64 (tolerance zero)."""
import numpy as np
import pytest

import oracle
from paper_2608_13696_gb300 import rel

from test_low_hints import L, hint_plan  # noqa: F401 (a fixture)

OPS = {2: ("sum", "count"), 4: ("sum", "count", "min", "max")}


@pytest.mark.parametrize("na", [2, 4])
@pytest.mark.parametrize("hint,n,bits,slots", [
    (90_000, 1 << 20, 7, 1 << 18), (90_000, (8000 << 7) - 1, 7, 1 << 16),  # pieces, whole
    (190_000, 8000 << 8, 8, 1 << 19), (190_000, 600_000, 8, 1 << 16),
    (250_000, 8000 << 8, 8, 1 << 19), (250_000, 600_000, 9, 1 << 16)])
def test_plan_follows_the_rows(L, na, hint, n, bits, slots):  # noqa: F811
    p = hint_plan(L, OPS[na], rel.I64, hint, n)
    assert (p.part_bits, p.slots) == (bits, slots)


@pytest.mark.gpu
@pytest.mark.parametrize("na", [2, 4])
@pytest.mark.parametrize("sketch", [0, rel.PLAN_SKETCH])
@pytest.mark.parametrize("kind", ["flat", "skewed"])
@pytest.mark.parametrize("n,groups", [(20_001, 6000), (127_999, 6000), (128_000, 6000), (700_003, 40_000)])
def test_results_on_both_sides(na, sketch, kind, n, groups):
    from gpu_util import canon_groupby, query_to_cuda

    rng = np.random.default_rng(n + na)
    r = rng.integers(0, groups, n)
    if kind == "skewed":
        r[rng.random(n) < 0.4] = 5
    v = rng.integers(-(2**62), 2**62, n)  # sums wrap
    q = oracle.kv_query(r * np.int64(1_000_003) - 7, v, ops=OPS[na])
    qc = query_to_cuda(q)
    p = rel.plan_groupby(qc, groups_hint=groups, flags=sketch | rel.plan_force(rel.VAR_PARTITIONED))
    assert (p.n_hot > 0) == (bool(sketch) and kind == "skewed")
    k, a = canon_groupby(*rel.groupby(qc, plan=p))
    ek, ea = oracle.groupby(q)
    np.testing.assert_array_equal(k, ek)
    np.testing.assert_array_equal(a, ea)


@pytest.mark.gpu
@pytest.mark.parametrize("na", [2, 4])
def test_low_hint_with_doubled_tables(na):
    """Equal pieces, tables twice the planned size (many rows per partition), and
    nearly twice the groups that were expected: they meet in the global table,
    which has the planned slots."""
    from gpu_util import canon_groupby, query_to_cuda

    n, hint, groups = 128 * 16384 + 5, 60_000, 115_000
    rng = np.random.default_rng(na)
    q = oracle.kv_query(rng.integers(0, groups, n) * 31, rng.integers(-99, 99, n), ops=OPS[na])
    qc = query_to_cuda(q)
    p = rel.plan_groupby(qc, groups_hint=hint)
    assert (p.part_bits, p.smem_slots, p.slots) == (7, 1024, 1 << 17)
    k, a = canon_groupby(*rel.groupby(qc, plan=p, capacity=groups))
    ek, ea = oracle.groupby(q)
    np.testing.assert_array_equal(k, ek)
    np.testing.assert_array_equal(a, ea)
