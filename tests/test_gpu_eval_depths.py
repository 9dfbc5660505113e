"""dc_eval_timeline_batch above 64 layers (one warp per instance, 64 rows at a time; one
thread on large batches of up to 257) against the oracle's event replay: odd and even
depths around the chunks, rows off a 16-byte boundary, no break, every break, ties, values
beyond 32 bits and faulty inputs."""
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


@pytest.mark.parametrize("copies", [1, 400])
@pytest.mark.parametrize("L", [65, 66, 95, 96, 127, 128, 129, 192, 193, 1025, 4096])
def test_replays_of_any_decision(dc, L, copies):
    import torch
    if copies > 1 and L > 96:
        pytest.skip("one kernel for every batch")
    B = 131
    comp, xfer, dt = wl.skewed_instances(7 + L, B, L)
    c2, x2, d2 = wl.tie_heavy_instances(L, 20, L)
    comp[:20], xfer[:20], dt[:20] = c2, x2, d2
    comp[20:40] <<= 20
    xfer[25:45] <<= 18
    comp[50, L - 1] = -1
    xfer[51, 64] = -1
    xfer[52, 0] = 1 << 52
    dt[53], dt[54] = -1, 1 << 52
    dt[55] = (1 << 52) // L + 1
    bits = np.concatenate([wl.random_decisions(L, 43, L, density=p) for p in (0.02, 0.4, 1.0)]
                          + [wl.random_decisions(L, 2, L, density=0.0)])
    for offset in (0, 1):  # 1: 8 bytes past a 16-byte boundary

        def dev(a):
            t = torch.from_numpy(np.ascontiguousarray(np.tile(a, (copies,) + (1,) * (a.ndim - 1))))
            buf = torch.empty(t.numel() + offset, dtype=t.dtype, device="cuda")
            buf[offset:].copy_(t.flatten())
            return buf[offset:].view(t.shape)
        for d in (0, 1):
            got = dc.eval_timeline(d, dev(comp), dev(xfer), dev(dt), dev(bits.view(np.int32)))
            exp = oracle.replay_batch(d, comp, xfer, dt, bits, nthreads=os.cpu_count() or 1)
            assert (got.cpu().numpy().reshape(copies, B) == exp[None]).all(), (L, d, offset)


@pytest.mark.parametrize("batch", [20_000, 40_000, 50_000, 80_000, 150_001])
@pytest.mark.parametrize("L", [65, 70, 72, 97, 100, 101, 112, 129, 131, 140, 142, 257, 259])
def test_where_a_thread_takes_an_instance(dc, L, batch):
    """Batches and depths on both sides of every line between a warp and a thread per
    instance."""
    import torch
    B = 125
    comp, xfer, dt = wl.skewed_instances(L, B, L)
    comp[:30] <<= 20
    xfer[50, L - 1], dt[51] = -1, 1 << 52
    bits = np.concatenate([wl.random_decisions(L, 60, L, density=0.1), wl.random_decisions(L, 65, L, density=0.9)])
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (comp, xfer, dt, bits.view(np.int32))]
    copies = -(-batch // B)
    for n in (batch - 1, batch):
        dev = [a.repeat((copies,) + (1,) * (a.dim() - 1))[:n].contiguous() for a in t]
        for d in (0, 1):
            exp = oracle.replay_batch(d, comp, xfer, dt, bits, nthreads=os.cpu_count() or 1)
            got = dc.eval_timeline(d, *dev).cpu().numpy()
            assert np.array_equal(got, np.tile(exp, copies)[:n]), (L, n, d)
