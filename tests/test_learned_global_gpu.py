"""A network that prefers the global table: followed as it is where one key is
as good as another and the input cannot be partitioned; elsewhere the rule by
group count chooses.  The estimate and the result do not depend on it."""
import numpy as np
import pytest
import torch

import oracle
from oracle import mlp as M
from paper_2608_13696_gb300 import rel

from gpu_util import canon_groupby, query_to_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ops", [("sum",), ("sum", "count")])
@pytest.mark.parametrize("kind", ["flat", "skewed"])
@pytest.mark.parametrize("flags", [rel.PLAN_LEARNED, rel.PLAN_LEARNED | rel.PLAN_SKETCH])
def test_preferred_global_table(ops, kind, flags):
    rng = np.random.default_rng(3)
    n, groups = 20_000, 6000
    r = rng.integers(0, groups, n)
    if kind == "skewed":
        r[rng.random(n) < 0.5] = 1
    q = oracle.kv_query(r * 977, rng.integers(-50, 50, n), ops=ops)
    p = np.zeros(M.N_PARAMS, np.float32)
    p[M.OFF_B3:] = [14.0, 0.0, 5.0, 0.0]  # log2 of the groups, then the variants
    rel.planner_set(torch.from_numpy(p).cuda())
    keys, aggs, plan = rel.groupby_auto(query_to_cuda(q), flags=flags)
    assert plan.est_groups == n  # 1.25 x 2^15, at most the rows
    if len(ops) == 2:  # key/value with sum and count: can be partitioned
        assert plan.variant == rel.VAR_PARTITIONED
    else:
        assert plan.variant == rel.VAR_GLOBAL
        assert plan.smem_slots == (2048 if kind == "skewed" else 0)
    k, a = canon_groupby(keys, aggs)
    ek, ea = oracle.groupby(q)
    np.testing.assert_array_equal(k, ek)
    np.testing.assert_array_equal(a, ea)
