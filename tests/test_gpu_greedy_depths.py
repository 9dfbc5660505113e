"""The greedy schedulers of one instance per warp (L <= 64) and per CTA at depths around
their warp, row-pair and search boundaries, in 32 and in 64 bits, and on both sides of the
lines to the kernel of one instance per thread, against the oracle; above L = 600, where
the oracle's backward enumeration is too slow, against the same rule by bisection."""
import bisect
import os

import numpy as np
import pytest

import oracle
from paper_2101_07968_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2101_07968_gb300 import build, dynacomm
    build.build()
    dynacomm.lib()
    return dynacomm


def _run(dc, d, comp, xfer, dt):
    import torch
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    out = dc.greedy(d, t(comp), t(xfer), t(dt))
    return out["makespan"].cpu().numpy(), out["bits"].cpu().numpy().view(np.uint32)


def _instances(L, B, wide):
    comp, xfer, dt = wl.skewed_instances(91 + L, B, L)
    comp[::4] = 0                      # no compute at all: every position ties
    comp[1::4, L // 3:] = 0            # a zero-compute tail and head
    if wide:
        comp[2::4] <<= 20
        xfer[::2] <<= 18
    return comp, xfer, dt


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("L", list(range(9, 19)) + [33, 34, 63, 64, 65, 66, 127, 128, 129, 257])
def test_depths(dc, L, wide):
    comp, xfer, dt = _instances(L, 21, wide)
    for d in (0, 1):
        mk, bits = _run(dc, d, comp, xfer, dt)
        exp = oracle.greedy_batch(d, comp, xfer, dt, nthreads=os.cpu_count() or 1)
        assert np.array_equal(mk, exp["makespan"]) and np.array_equal(bits, exp["bits"]), (L, d)


def _backward(bc, gt, dt):
    """Algorithm 2 in processing order: every first push p, each next segment as long
    as the link estimate covers, least f_m, the longest first push on ties."""
    A, B = [0], [0]
    for c, x in zip(bc[::-1].tolist(), gt[::-1].tolist()):
        A.append(A[-1] + c)
        B.append(B[-1] + x)
    L, best = len(bc), None
    for p0 in range(L - 1, 0, -1):
        p, sent, link, cuts = p0, dt, A[p0] + dt + B[p0], []
        while p < L:
            cuts.append(p)
            q = bisect.bisect_right(A, max(A[p] + sent + B[p], A[p + 1])) - 1
            link = max(link, A[q]) + dt + B[q] - B[p]
            p, sent = q, sent + dt
        if best is None or link < best[0]:
            best = (link, cuts)
    return best


@pytest.mark.parametrize("L", [600, 1025, 2049])
def test_deep(dc, L):
    comp, xfer, dt = _instances(L, 5, True)
    mk, bits = _run(dc, 0, comp, xfer, dt)
    if L <= 1025:  # the oracle enumerates every pair
        exp = oracle.greedy_batch(0, comp, xfer, dt, nthreads=os.cpu_count() or 1)
        assert np.array_equal(mk, exp["makespan"]) and np.array_equal(bits, exp["bits"])
    else:
        assert np.array_equal(mk, oracle.replay_batch(0, comp, xfer, dt, bits))
    mk, bits = _run(dc, 1, comp, xfer, dt)
    for i in range(len(dt)):
        t, cuts = _backward(comp[i], xfer[i], int(dt[i]))
        word = np.zeros(dc.words(L), np.uint32)
        for q in cuts:
            word[(q - 1) // 32] |= np.uint32(1 << ((q - 1) % 32))
        assert mk[i] == t and np.array_equal(bits[i], word), (L, i)


def _edge_instances(L, total):
    """Sums of a[L] + b[L] + (L + 1) dt = total, with and without a zero-cost tail in
    processing order of either direction, concentrated in a layer or spread."""
    rng = np.random.default_rng(L)
    comp, xfer, dt = [], [], []
    for d in (0, 1, 1 << 20):
        rest = total - (L + 1) * d
        for j in (0, 1, L // 2, L - 1):  # layers below j (or above L - 1 - j) cost nothing
            for x in (0, 1, rest // 2, rest):
                c, t = np.zeros(L, np.int64), np.zeros(L, np.int64)
                c[j], t[j] = rest - x, x
                spread = np.diff(np.r_[0, np.sort(rng.integers(0, rest + 1, 2 * (L - j) - 1)), rest])
                cs, ts = np.zeros(L, np.int64), np.zeros(L, np.int64)
                cs[j:], ts[j:] = spread[::2], spread[1::2]
                for a, b in ((c, t), (c, t[::-1]), (cs, ts)):
                    comp += [a, a[::-1]]
                    xfer += [b, b[::-1]]
                    dt += [d, d]
    return np.array(comp), np.array(xfer), np.array(dt, np.int64)


@pytest.mark.parametrize("total", [2**31 - 2, 2**31 - 1, 2**31])
@pytest.mark.parametrize("L", [8, 9, 16, 22, 23, 33, 63, 64, 65, 129])
def test_sums_at_two_to_the_31(dc, L, total):
    """The 32-bit forms end at a sum of 2^31 - 1, where no value may grow by one more."""
    comp, xfer, dt = _edge_instances(L, total)
    for d in (0, 1):
        mk, bits = _run(dc, d, comp, xfer, dt)
        exp = oracle.greedy_batch(d, comp, xfer, dt, nthreads=os.cpu_count() or 1)
        assert np.array_equal(mk, exp["makespan"]) and np.array_equal(bits, exp["bits"]), (L, d)


# 5,001: four warps to a CTA, several instances to a warp; from 50,000 and 100,000 on some
# depths take a thread per instance
@pytest.mark.parametrize("batch", [5_001, 49_999, 50_000, 99_999, 100_000])
@pytest.mark.parametrize("L", [8, 9, 12, 13, 16, 22, 23, 24, 25, 27, 54, 64, 65, 128, 129])
def test_large_batches(dc, L, batch):
    import torch
    comp, xfer, dt = _instances(L, 41, False)
    comp[20:31] <<= 22  # mixed widths within a warp's and a CTA's instances
    xfer[25:36] <<= 20
    comp[37, L - 1], xfer[38, 0], dt[39] = -1, 1 << 52, -4  # faults between good ones
    copies = -(-batch // len(dt))
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda().repeat((copies,) + (1,) * (a.ndim - 1))[:batch]
         .contiguous() for a in (comp, xfer, dt)]
    for d in (0, 1):
        out = dc.greedy(d, *t)
        exp = oracle.greedy_batch(d, comp, xfer, dt, nthreads=os.cpu_count() or 1)
        assert np.array_equal(out["makespan"].cpu().numpy(), np.tile(exp["makespan"], copies)[:batch]), (L, d)
        assert np.array_equal(out["bits"].cpu().numpy().view(np.uint32),
                              np.tile(exp["bits"], (copies, 1))[:batch]), (L, d)
