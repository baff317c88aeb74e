"""Calls whose kernels take different amounts of shared memory do not disturb
one another: a kernel's limit is the same for all of them, so neither another
batch nor another host thread's smaller plan can take it below what a launch
needs.  Results are exact int64 (tolerance zero)."""
import ctypes
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_2608_13696_gb300 import rel

from gpu_util import canon_groupby, cuda, query_to_cuda

pytestmark = pytest.mark.gpu
OPS = ("sum", "count", "min", "max")
CALLS = 2000


def table(n, groups, seed):
    rng = np.random.default_rng(seed)
    return rng.integers(0, groups, n) * 7919 - 5, rng.integers(-10**6, 10**6, n)


def test_a_small_batch_prepared_after_a_large_one():
    def batch(groups, n, cfg):
        k, v = table(n, groups, groups)
        b = rel.Batch([{"keys": cuda(k), "vals": cuda(v), "ops": list(OPS),
                        "slots": 1 << (2 * groups - 1).bit_length(), "est_groups": groups,
                        "capacity": groups}], []).prepare(cfg)
        return b, oracle.groupby(oracle.kv_query(k, v, ops=OPS))

    large, exp = batch(2000, 30_011, (256, 8, 1, 2048))
    small, exp_s = batch(8, 5_003, (256, 8, 1, 2048))
    for b, e in ((large, exp), (small, exp_s), (large, exp)):
        b.run()
        counts, flags = b.results()
        assert not any(flags)
        k, a = canon_groupby(*b.groupby_output(0, counts[0]))
        np.testing.assert_array_equal(k, e[0])
        np.testing.assert_array_equal(a, e[1])


@pytest.mark.parametrize("agg_count", [4, 1])
@pytest.mark.parametrize("hints", [(8, 2500), (700, 5000), (100, 60_000)])
def test_two_threads_with_different_plans(agg_count, hints):
    """Shared tables of several sizes and partitioned plans (four aggregates),
    the descriptor-driven kernel (one aggregate)."""
    jobs = []
    for h in hints:
        k, v = table(20_011, h, h)
        q = oracle.kv_query(k, v, ops=OPS[:agg_count])
        qc = query_to_cuda(q)
        jobs.append((qc, rel.plan_groupby(qc, groups_hint=h), oracle.groupby(q)))
    torch.cuda.synchronize()
    wrong, L = [], rel.load()

    def work(qc, plan, exp):
        try:
            d = rel._Desc(qc)
            ws = rel._ws(plan.workspace_bytes, "cuda")
            cap = len(exp[0])
            out = torch.empty((1 + agg_count, cap), dtype=torch.int64, device="cuda")
            ptrs = (ctypes.c_void_p * agg_count)(*[out[1 + a].data_ptr() for a in range(agg_count)])
            s = torch.cuda.Stream()
            for i in range(CALLS):  # launches only, but for the last
                n = ctypes.c_int64(0)
                rel._check(L.rel_groupby_agg(
                    ctypes.byref(d.d), ctypes.byref(plan), ws.data_ptr(), ws.numel(), out[0].data_ptr(),
                    ptrs, cap, ctypes.byref(n) if i == CALLS - 1 else None, s.cuda_stream))
            got = canon_groupby(out[0][:n.value], list(out[1:, :n.value]))
            if not (np.array_equal(got[0], exp[0]) and np.array_equal(got[1], exp[1])):
                wrong.append("results differ")
        except Exception as e:  # noqa: BLE001 (reported below)
            wrong.append(str(e))

    ts = [threading.Thread(target=work, args=j) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not wrong, wrong[0]
