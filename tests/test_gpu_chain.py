"""The CTA-per-instance solver (first pass above L = 256, work lists below) where it
can go wrong: depths around its row-pair, warp and search boundaries, optima around
the last column it keeps, values that do not fit its 32-bit kept offsets, and inputs
that make every column tie. Bit for bit against the oracle."""
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


def _same(dc, comp, xfer, dt, label):
    import torch
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    W, out = dc.words(comp.shape[1]), {}
    for d in (0, 1):
        got = {k: v.cpu().numpy() for k, v in dc.schedule(d, t(comp), t(xfer), t(dt)).items()}
        exp = oracle.schedule_batch(d, comp, xfer, dt, nthreads=os.cpu_count() or 1)
        for k in ("status", "makespan", "nseg"):
            assert np.array_equal(got[k], exp[k]), (label, d, k)
        assert np.array_equal(got["bits"].view(np.uint32)[:, :W], exp["bits"]), (label, d)
        out[d] = exp["nseg"]
    return out


@pytest.mark.parametrize("L", [257, 259, 511, 512, 513, 514, 767])
def test_depths_around_the_boundaries(dc, L):
    """Two rows per thread, 8 per warp lane, powers of two of the search: odd and even
    depths on both sides, with values beyond 32 bits among them."""
    comp, xfer, dt = wl.skewed_instances(61 + L, 24, L)
    comp[::3] <<= 18
    xfer[1::3] <<= 16
    _same(dc, comp, xfer, dt, L)


@pytest.mark.parametrize("L", [40, 300])
def test_optima_around_the_last_kept_column(dc, L):
    """Equal layers and a latency from 0 up: from L segments down to a few, on both
    sides of the 9 (L = 40) and 65 (L = 300) segments the first pass traces back."""
    B = 48
    comp = np.full((B, L), 1000, dtype=np.int64)
    xfer = np.full((B, L), 990, dtype=np.int64)
    dt = np.arange(B, dtype=np.int64) * (6 if L == 300 else 40)
    s = _same(dc, comp, xfer, dt, L)
    limit = 65 if L == 300 else 9
    assert any((s[d] > limit).any() and (s[d] <= limit).any() for d in (0, 1))


@pytest.mark.parametrize("L", [20, 70, 300])
def test_values_spanning_more_than_32_bits(dc, L):
    """Idle time and push backlog of more than 2^32 us: whole 64-bit values."""
    comp, xfer, dt = wl.random_instances(5 + L, 30, L, 1 << 30, 1 << 38, 1 << 20, 1 << 34)
    comp[::2] >>= 9
    xfer[1::3] >>= 8
    _same(dc, comp, xfer, dt, L)


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
