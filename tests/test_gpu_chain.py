"""The chain solver of 17 layers and more (a warp per instance up to 192, a CTA above, and
their work lists) where it can go wrong: depths around its row-pair, warp and search
boundaries, optima around the last column a pass keeps, values that do not fit its
32-bit kept offsets, and inputs that make every column tie. Bit for bit against the
oracle."""
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


def _same(dc, comp, xfer, dt, label, copies=1):
    """Both directions of the instances, repeated `copies` times. Returns per direction
    the oracle's segment counts and how many instances the first pass listed (a batch
    that one launch solves lists none)."""
    import torch
    t = lambda a: (torch.from_numpy(np.ascontiguousarray(a)).cuda()
                   .repeat((copies,) + (1,) * (a.ndim - 1)))
    B, L = comp.shape
    sched, out = dc.Scheduler(copies * B, L), {}
    for d in (0, 1):
        got = {k: v.cpu().numpy() for k, v in sched.run(d, t(comp), t(xfer), t(dt)).items()}
        exp = oracle.schedule_batch(d, comp, xfer, dt, nthreads=os.cpu_count() or 1)
        for k in ("status", "makespan", "nseg"):
            assert np.array_equal(got[k], np.tile(exp[k], copies)), (label, d, k)
        assert np.array_equal(got["bits"].view(np.uint32)[:, :dc.words(L)],
                              np.tile(exp["bits"], (copies, 1))), (label, d)
        out[d] = exp["nseg"], int(sched.workspace[:4].view(torch.int32))
    return out


@pytest.mark.parametrize("L", [257, 259, 511, 512, 513, 514, 767])
def test_depths_around_the_boundaries(dc, L):
    """Two rows per thread, 8 per warp lane, powers of two of the search: odd and even
    depths on both sides, with values beyond 32 bits among them."""
    comp, xfer, dt = wl.skewed_instances(61 + L, 24, L)
    comp[::3] <<= 18
    xfer[1::3] <<= 16
    _same(dc, comp, xfer, dt, L)


# the batch is repeated to at least this many, and the first pass traces back optima of up to
# `limit` segments: thread per instance, warp (two, four, six rows per lane), CTA
@pytest.mark.parametrize("L,least,limit", [(18, 160_000, 9), (40, 41_000, 25), (100, 1, 25),
                                           (160, 1, 25), (200, 1, 65), (300, 1, 65)])
def test_optima_around_the_last_kept_column(dc, L, least, limit):
    """Equal layers and a latency from 0 up: from L segments down to a few, on both sides
    of the columns that lie in shared memory (8 of a warp) and of the last one kept; what
    needs more is listed, and nothing else."""
    dt = np.unique(np.r_[np.arange(0, 60), np.round(np.geomspace(60, 20000, 240))]).astype(np.int64)
    comp = np.full((len(dt), L), 1000, dtype=np.int64)
    xfer = np.full((len(dt), L), 990, dtype=np.int64)
    copies = -(-least // len(dt))
    assert dc.dc_schedule_kernel_launches(copies * len(dt), L) == 2
    for d, (s, listed) in _same(dc, comp, xfer, dt, L, copies).items():
        assert {8, 9, 10, limit - 1, limit, limit + 1} <= set(s.tolist()), d
        assert listed == copies * int((s > limit).sum()), d


@pytest.mark.parametrize("copies", [1, 700])
@pytest.mark.parametrize("L", [65, 66, 127, 128, 129, 191, 192, 193, 194, 256])
def test_warp_and_cta_depths(dc, L, copies):
    """Every count of rows per lane, full and one row over, and the first depths of the CTA
    form; once few instances, once (up to 192) enough that the warps take a share of their
    own and then runs from the ticket."""
    if copies > 1 and L > 192:
        pytest.skip("a CTA takes one instance at a time")
    parts = [wl.skewed_instances(L, 70, L), wl.tie_heavy_instances(L, 30, L), wl.skewed_instances(L + 1, 31, L)]
    comp, xfer, dt = (np.concatenate([p[q] for p in parts]) for q in range(3))
    comp[100:] <<= 18
    xfer[90:120] <<= 16
    comp[3, L - 1], xfer[4, 64], dt[5] = -1, 1 << 52, -3
    _same(dc, comp, xfer, dt, (L, copies), copies)


@pytest.mark.parametrize("L,least", [(20, 1), (20, 41_000), (70, 1), (300, 1)])
def test_values_spanning_more_than_32_bits(dc, L, least):
    """Idle time and push backlog of more than 2^32 us: whole 64-bit values, in a pass that
    keeps them all or, where it keeps 32-bit words, listed."""
    comp, xfer, dt = wl.random_instances(5 + L, 30, L, 1 << 30, 1 << 38, 1 << 20, 1 << 34)
    comp[::2] >>= 9
    xfer[1::3] >>= 8
    copies = -(-least // 30)
    one = dc.dc_schedule_kernel_launches(copies * 30, L) == 1
    for d, (_, listed) in _same(dc, comp, xfer, dt, L, copies).items():
        assert (listed == 0) == one, d


@pytest.mark.parametrize("L", [33, 129, 400])
@pytest.mark.parametrize("zero", ["comp", "xfer", "dt", "all"])
def test_ties_everywhere(dc, L, zero):
    """Zero costs or latency: every split ties, the lowest split and the fewest
    segments have to win."""
    comp, xfer, dt = wl.random_instances(L, 40, L, 0, 1, 0, 2)
    for name, a in (("comp", comp), ("xfer", xfer), ("dt", dt)):
        if zero in (name, "all"):
            a[:] = 0
    _same(dc, comp, xfer, dt, (L, zero))


@pytest.mark.parametrize("L", [639, 640, 641, 1023, 1024, 1025])
def test_searches_from_the_last_columns_end(dc, L):
    """From 640 layers on a search starts where the last column's ended: crossings that
    stay, that move a little, and that jump (one layer as long as hundreds), near both
    ends of the keys, with many columns and values beyond 32 bits among them."""
    parts = [wl.skewed_instances(L, 10, L), wl.tie_heavy_instances(L + 1, 6, L)]
    rng = np.random.default_rng(L)
    comp = rng.integers(1, 2000, (16, L))
    xfer = rng.integers(1, 2000, (16, L))
    for i in range(16):
        comp[i, rng.integers(0, L, 4)] *= 10 ** (i % 4)
        xfer[i, rng.integers(0, L, 4)] *= 10 ** (i // 4)
    comp[:4, : L // 2] = 0
    xfer[4:8, L // 2:] = 0
    comp[8:12] <<= 22
    xfer[8:12] <<= 22
    dt = rng.integers(0, 4000, 16)
    dt[8:12] <<= 22
    parts.append((comp.astype(np.int64), xfer.astype(np.int64), dt.astype(np.int64)))
    _same(dc, *(np.concatenate([p[q] for p in parts]) for q in range(3)), L)
