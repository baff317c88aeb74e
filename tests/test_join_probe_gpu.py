"""Join probes at the sizes where the probe kernels change their course: rows
per thread by size (one up to 16 CTA rounds of the chip, two above), ragged
tails, probe columns off 16-byte alignment,
unique and repeated build keys, warps with many times the buffered matches,
INT64_MIN on both sides, outputs that are too small.  Whole numbers: exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_13696_gb300 import rel

from gpu_util import canon_join, cuda

pytestmark = pytest.mark.gpu
MIN = np.iinfo(np.int64).min


def sides(nb, npr, per_key, side, seed):
    rng = np.random.default_rng(seed)
    bk = np.repeat(rng.permutation(4 * nb)[: -(-nb // per_key)], per_key)[:nb].astype(np.int64)
    bk = rng.permutation(bk * 0x1000003 - 77)
    pk = np.where(rng.random(npr) < 0.7, bk[rng.integers(0, nb, npr)],
                  rng.integers(-(2**62), 2**62, npr)).astype(np.int64)
    if side:
        bk[:: max(1, nb // 3)] = MIN
        pk[:: max(1, npr // 40)] = MIN
    return bk, rng.integers(-(2**63), 2**63 - 1, nb, dtype=np.int64), pk


SMALL = 152 * 4 * 256 * 4  # above: more rows per thread (on 152 SMs)


@pytest.mark.parametrize("nb,npr,per_key,side", [
    (1, 1, 1, False), (7, 255, 1, True), (500, 257, 3, True), (40, 3001, 40, False),
    (300, 1025, 300, False), (1000, SMALL, 1, True), (1000, SMALL + 1, 1, False),
    (5000, SMALL + 511, 2, True), (65536, SMALL + 2047, 1, True), (90, SMALL + 5, 3, False)])
@pytest.mark.parametrize("off", [0, 1])
def test_probe_course(nb, npr, per_key, side, off):
    bk, bp, pk = sides(nb, npr, per_key, side, seed=nb + npr)
    t = rel.JoinTable(cuda(bk), cuda(bp))
    pkc = cuda(np.concatenate([np.zeros(off, np.int64), pk]))[off:]
    epi, ebi, epay = oracle.join(bk, bp, pk)
    assert t.count(pkc) == len(epi)
    pi, bi, pay = canon_join(*t.probe(pkc, capacity=max(1, len(epi))))
    np.testing.assert_array_equal(pi, epi)
    np.testing.assert_array_equal(bi, ebi)
    np.testing.assert_array_equal(pay, epay)


@pytest.mark.parametrize("npr", [3001, SMALL + 511])
def test_short_outputs_hold_true_pairs(npr):
    """A short output is refused with the true count, and nothing is written past it."""
    import ctypes
    bk, bp, pk = sides(700, npr, 2, True, seed=5)
    t = rel.JoinTable(cuda(bk), cuda(bp))
    pkc = cuda(pk)
    cap, want = 777, len(oracle.join(bk, bp, pk)[0])
    pi = torch.full((cap + 64,), -5, dtype=torch.int32, device="cuda")
    bi, pay = pi.clone(), torch.full((cap + 64,), -5, dtype=torch.int64, device="cuda")
    n = ctypes.c_int64(0)
    L = rel.load()
    r = L.rel_join_probe(ctypes.byref(t.t), pkc.data_ptr(), npr, pi.data_ptr(), bi.data_ptr(),
                         pay.data_ptr(), cap, ctypes.byref(n),
                         torch.cuda.current_stream().cuda_stream)
    assert r == rel.REL_E_CAPACITY and n.value == want
    torch.cuda.synchronize()
    assert bool((pi[cap:] == -5).all()) and bool((bi[cap:] == -5).all())
    assert bool((pay[cap:] == -5).all())
    p, b = pi[:cap].cpu().numpy(), bi[:cap].cpu().numpy()
    assert (bk[b] == pk[p]).all() and (bp[b] == pay[:cap].cpu().numpy()).all()


@pytest.mark.parametrize("n", [2, 3, 1000, 4097, 262_144])
@pytest.mark.parametrize("copies", [1, 2, 3, 64])
def test_build_with_repeated_keys(n, copies):
    """Copies of a key claim the slots behind its first one, in pairs that fill
    up; one repeated key among different ones is noticed."""
    rng = np.random.default_rng(n + copies)
    bk = np.arange(n, dtype=np.int64) // copies * 7919 - n
    if copies == 1:
        bk[-1] = bk[0]
    bk = bk[rng.permutation(n)]
    bp = rng.integers(0, 2**62, n)
    pk = np.concatenate([np.unique(bk), np.unique(bk)[:5] + 1])
    e = oracle.join(bk, bp, pk)
    t = rel.JoinTable(cuda(bk), cuda(bp))
    assert t.count(cuda(pk)) == len(e[0]) == n
    for x, y in zip(canon_join(*t.probe(cuda(pk), capacity=n)), e):
        np.testing.assert_array_equal(x, y)
