"""The exact count with a sketch beside it: the key set keeps its full size (a
set of half the slots is full when every key is another, and the count then
walks it to its end and starts again), and a count that does start again keeps
the sketch taken with its first attempt."""
import ctypes

import pytest
import torch

from paper_2608_13696_gb300 import rel

pytestmark = pytest.mark.gpu
BOTH = rel.PLAN_EXACT | rel.PLAN_SKETCH


def packed(n):
    """n different (uint8, int32) keys and one value column."""
    i = torch.arange(n, device="cuda")
    return {"cols": [(i % 5).to(torch.uint8), (i // 5).to(torch.int32), i.clone()], "keys": [0, 1],
            "preds": [], "aggs": [("sum", 2, []), ("min", 2, [])]}


@pytest.mark.parametrize("n", [8192, 2**18 - 1, 2**18, 2**18 + 1])
def test_every_key_another(n):
    q = packed(n)
    rel.plan_groupby(q, flags=BOTH)
    n0 = rel.launch_count()
    p = rel.plan_groupby(q, flags=BOTH)
    assert p.est_groups == n
    assert rel.launch_count() - n0 == 2  # sketch and count, once each


def test_workspace_without_room_for_the_sketch():
    """What held the key set alone is still enough: the sketch comes after."""
    n = 8192
    q = packed(n)
    d = rel._Desc(q)
    need = 256 + 8 * 2 * n
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    p = rel.Plan()
    args = (rel.OP_GROUPBY, ctypes.byref(d.d), BOTH, 0, ws.data_ptr())
    rel._check(rel.load().rel_plan_size(*args, need, ctypes.byref(p), None))
    assert p.est_groups == n and p.scratch_bytes <= need
    assert rel.load().rel_plan_size(*args, need - 1, ctypes.byref(p), None) == rel.REL_E_CAPACITY


def test_sketch_survives_a_second_count():
    """More keys than the first set holds, and one in a tenth of the rows."""
    n, hot = 36_000_000, 123_456_789_012_345
    k = torch.cat([torch.arange(n, device="cuda") * 1_000_003, torch.full((n // 9,), hot, device="cuda")])
    k = k.view(10, n // 9).t().reshape(-1)  # the hot key in every tenth row
    q = {"cols": [k.contiguous(), k], "keys": [0], "preds": [], "aggs": [("sum", 1, []), ("count", 1, [])]}
    n0 = rel.launch_count()
    p = rel.plan_groupby(q, flags=BOTH)
    assert rel.launch_count() - n0 > 2
    assert p.est_groups == n + 1
    assert hot in [p.hot_keys[i] for i in range(p.n_hot)]
