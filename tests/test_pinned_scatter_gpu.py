"""Pinned keys in the partitioned passes: their thread-private words, for one
pinned key up to as many as a plan has, int32 and int64 keys, two and four
aggregates, extreme values (32-bit counts, min and max stored only on change,
sums that wrap), ragged sizes.  Whole numbers: exact."""
import numpy as np
import pytest

from paper_2608_13696_gb300 import rel, workloads

from gpu_util import cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hot", [1, 3, 8])
@pytest.mark.parametrize("kt", ["int64", "int32"])
@pytest.mark.parametrize("ops", [("sum", "count"), ("sum", "count", "min", "max")])
def test_pinned_partitions(hot, kt, ops):
    rng = np.random.default_rng(hot)
    n = 1_000_003 + hot
    k = rng.integers(-200_000, 200_000, n).astype(kt)
    is_hot = rng.random(n) < 0.5
    k[is_hot] = (7 * rng.integers(0, hot, n) - 3).astype(kt)[is_hot]
    v = rng.integers(-(2**63), 2**63 - 1, n, dtype=np.int64)
    v[:4] = [2**63 - 1, -(2**63), -1, 0]
    q = workloads.kv_query(cuda(k), cuda(v), list(ops))
    plan = rel.plan_groupby(q, flags=rel.PLAN_SKETCH | rel.plan_force(3), groups_hint=410_000)
    gk, ga = rel.groupby(q, plan=plan)
    keys, inv = np.unique(k.astype(np.int64), return_inverse=True)
    order = np.argsort(gk.cpu().numpy())
    np.testing.assert_array_equal(gk.cpu().numpy()[order], keys)
    want = {"sum": np.zeros(len(keys), np.int64), "count": np.bincount(inv),
            "min": np.full(len(keys), 2**63 - 1), "max": np.full(len(keys), -(2**63))}
    np.add.at(want["sum"], inv, v)
    np.minimum.at(want["min"], inv, v)
    np.maximum.at(want["max"], inv, v)
    for op, a in zip(ops, ga):
        np.testing.assert_array_equal(a.cpu().numpy()[order], want[op])
