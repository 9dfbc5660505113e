"""The pass over the instances that the short-row passes (L <= 16) leave behind, values past
32 bits and optima deeper than the kept columns: lists on both sides of the line between a
warp and a lane per instance, that fill a round of lanes or leave a remainder, at the depths
where the form changes; against the oracle."""
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


def _batch(L, n, B):
    """B instances, n of which are listed: past 32 bits, every other one without latency
    (as many segments as pay), spread over the batch; the others need few segments."""
    rng = np.random.default_rng(L)
    comp = rng.integers(0, 1000, (B, L))
    xfer = rng.integers(0, 1000, (B, L))
    dt = rng.integers(4000, 9000, B)
    at = rng.permutation(B)[:n]
    comp[at] = rng.integers(0, 1 << rng.integers(33, 45, n)[:, None], (n, L))
    xfer[at] = rng.integers(0, 1 << rng.integers(33, 45, n)[:, None], (n, L))
    dt[at] = rng.integers(0, 1 << 32, n)
    dt[at[::2]] = 0
    comp[at[::3], : L // 2] = 0  # ties
    comp[at, L - 1] += 1 << 33
    return comp, xfer, dt.astype(np.int64)


@pytest.mark.parametrize("L", [1, 2, 4, 5, 6, 7, 8, 11, 12, 15, 16])
@pytest.mark.parametrize("n", [1, 1200, 1201, 2432, 2433, 30_011])
def test_listed_instances(dc, L, n):
    import torch
    B = 30_011
    comp, xfer, dt = _batch(L, n, B)
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (comp, xfer, dt)]
    s = dc.Scheduler(B, L)
    replay = torch.empty(B, dtype=torch.int64, device="cuda")
    for d in (0, 1):
        exp = oracle.schedule_batch(d, comp, xfer, dt, nthreads=os.cpu_count() or 1)
        o = s.run(d, *t)
        assert int(s.workspace[:4].view(torch.int32)) == n
        plain = {k: v.clone() for k, v in o.items()}
        for v in o.values():
            v.fill_(-1)
        assert dc.dc_schedule_replay_batch(d, B, L, *t, o["makespan"], o["bits"], o["nseg"], o["status"],
                                           replay, s.workspace, s.ws_bytes) == dc.DC_OK
        for out in (plain, o):
            for k in ("makespan", "nseg", "status"):
                assert np.array_equal(out[k].cpu().numpy(), exp[k]), (k, d)
            if L > 1:
                assert np.array_equal(out["bits"].cpu().numpy().view(np.uint32), exp["bits"]), d
        assert torch.equal(replay, o["makespan"])


# rates of 1 to 100,000 FLOP/us leave a tenth of the instances or so past 32 bits
@pytest.mark.parametrize("L", [1, 4, 5, 8, 12, 13, 16])
@pytest.mark.parametrize("kw", [dict(rate_dist=1, rate_lo=1, flops_lo=1 << 30, flops_hi=1 << 32),
                                dict(rate_lo=1, rate_hi=1, flops_lo=3 << 30, flops_hi=1 << 33)])
def test_listed_draws(dc, L, kw):
    import torch
    B = 12_007
    cfg = wl.with_batch(wl.config("tiny"), B)
    cfg.update(L=L, **kw)
    cfg.update(dt_lo=0, dt_hi=1 << 20)
    prof = oracle.profile_gen(cfg)
    g = dc.GeneratedScheduler(cfg)
    out = g.run()
    count = g.ws[:8].view(torch.int32).cpu().numpy()
    assert (count == B).all() if "rate_dist" not in kw else ((count > 100) & (count <= 4864)).all(), count
    for d, (c, x) in ((0, ("fc", "pt")), (1, ("bc", "gt"))):
        exp = oracle.schedule_batch(d, prof[c], prof[x], prof["dt"], nthreads=os.cpu_count() or 1)
        for k in ("makespan", "nseg", "status"):
            assert np.array_equal(out[k][d].cpu().numpy(), exp[k]), (k, d)
        if L > 1:
            assert np.array_equal(out["bits"][d].cpu().numpy().view(np.uint32), exp["bits"]), d
