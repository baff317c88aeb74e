"""The fused filter + product-form group-by over more (uint8, uint8) groups than
stay thread-private, planned with and without a sketch or a count.  Exact int64:
the tolerance is zero."""
import numpy as np
import pytest

import oracle
import synth
from paper_2608_13696_gb300 import rel

from gpu_util import canon_groupby, query_to_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("groups", [(7, 1), (3, 3), (16, 16), (256, 250)])
@pytest.mark.parametrize("n", [40, 4097, 300_001])
@pytest.mark.parametrize("plan", [{"flags": rel.PLAN_EXACT}, {"groups_hint": 8},
                                  {"flags": rel.PLAN_EXACT | rel.PLAN_SKETCH}, {"flags": 0}])
def test_fused_shape_with_many_groups(groups, n, plan):
    rng = np.random.default_rng(n + groups[0])
    li = synth.lineitem(n, seed=n)
    li["flag"] = rng.integers(0, groups[0], n).astype(np.uint8)
    li["status"] = rng.integers(0, groups[1], n).astype(np.uint8)
    q = oracle.lineitem_query(li)
    if plan.get("groups_hint"):
        plan = {"groups_hint": max(1, len(oracle.groupby(q)[0]))}
    k, a = canon_groupby(*rel.groupby(query_to_cuda(q), **plan))
    ek, ea = oracle.groupby(q)
    np.testing.assert_array_equal(k, ek)
    np.testing.assert_array_equal(a, ea)
