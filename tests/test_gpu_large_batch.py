"""The passes that only large batches take (the dense and looped kernels, the warp kernel
with its tickets, and their work lists) on hard instances: ties, skewed costs, values
beyond 32 bits, optima of many segments and input faults, repeated to a batch above the
single-launch limits. Every copy has to come out like the oracle's."""
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


def _hard(L):
    parts = [wl.tie_heavy_instances(L, 150, L), wl.skewed_instances(L + 1, 150, L),
             wl.random_instances(L + 2, 60, L), wl.skewed_instances(L + 3, 40, L)]
    comp, xfer, dt = (np.concatenate([p[q] for p in parts]) for q in range(3))
    comp[-40::2] <<= 24          # 64-bit values
    xfer[-39::2] <<= 22
    comp[150:200] = 1000         # equal layers and hardly any latency: many segments
    xfer[150:200] = 990
    dt[150:200] = np.arange(50) // 2
    comp[7, L - 1] = -1
    xfer[300, 0] = 1 << 52
    dt[301] = -5
    return comp, xfer, dt


@pytest.mark.parametrize("L", list(range(1, 21)) + [31, 32, 33, 47, 54, 63, 64])
def test_hard_instances_repeated(dc, L):
    import torch
    comp, xfer, dt = _hard(L)
    copies = (170_000 if L in (17, 18, 19) else 41_000) // len(dt) + 1
    t = lambda a: torch.from_numpy(np.ascontiguousarray(np.tile(a, (copies,) + (1,) * (a.ndim - 1)))).cuda()
    W = dc.words(L)
    assert dc.dc_schedule_kernel_launches(copies * len(dt), L) == 2
    for d in (0, 1):
        out = dc.schedule(d, t(comp), t(xfer), t(dt))
        exp = oracle.schedule_batch(d, comp, xfer, dt, nthreads=os.cpu_count() or 1)
        for k in ("status", "makespan", "nseg"):
            got = out[k].cpu().numpy().reshape(copies, -1)
            assert (got == exp[k][None]).all(), (L, d, k)
        got = out["bits"].cpu().numpy().view(np.uint32)[:, :W].reshape(copies, len(dt), W)
        assert (got == exp["bits"].reshape(1, len(dt), W)).all(), (L, d)


@pytest.mark.parametrize("L", [1, 2, 3, 4, 5, 6, 7])
def test_short_rows_many_tiles(dc, L):
    """Several tiles to a warp, a ragged last one, odd rows copied by 8 bytes."""
    cfg = wl.lsweep_config(L, 400_017)
    prof = dc.profile_gen(cfg)
    W = dc.words(L)
    for d, (c, x) in ((0, ("fc", "pt")), (1, ("bc", "gt"))):
        out = dc.schedule(d, prof[c], prof[x], prof["dt"])
        exp = oracle.schedule_batch(d, *(prof[k].cpu().numpy() for k in (c, x, "dt")),
                                    nthreads=os.cpu_count() or 1)
        for k in ("status", "makespan", "nseg"):
            assert (out[k].cpu().numpy() == exp[k]).all(), (L, d, k)
        got = out["bits"].cpu().numpy().view(np.uint32)[:, :W]
        assert (got == exp["bits"].reshape(len(got), W)).all(), (L, d)
