"""dc_schedule_replay_batch against the separate calls and the oracle: the schedule's
outputs unchanged, and replay equal to f_m of the written decision, on every kernel that
evaluates it (one launch, dense, looped, warp and CTA passes, and their work lists)."""
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


@pytest.mark.parametrize("L,copies", [(1, 1), (1, 90), (2, 1), (7, 1), (8, 90), (13, 300), (16, 1),
                                      (16, 300), (17, 1800), (19, 1800), (33, 500), (54, 1),
                                      (54, 300), (100, 2), (190, 2), (257, 1), (600, 1)])
def test_replay_of_the_written_decision(dc, L, copies):
    import torch
    parts = [wl.tie_heavy_instances(L, 30, L), wl.skewed_instances(L + 1, 40, L),
             wl.skewed_instances(L + 2, 30, L)]
    comp, xfer, dt = (np.concatenate([p[q] for p in parts]) for q in range(3))
    comp[-30::2] <<= 22
    xfer[-29::2] <<= 24
    comp[35:45] = 1000           # many segments
    xfer[35:45] = 990
    dt[35:45] = np.arange(10)
    comp[3, 0] = -1
    xfer[50, L - 1] = 1 << 52
    comp, xfer, dt = (np.tile(a, (copies,) + (1,) * (a.ndim - 1)) for a in (comp, xfer, dt))
    B, W = len(dt), dc.words(L)
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (comp, xfer, dt)]
    for d in (0, 1):
        ref = {k: v.clone() for k, v in dc.schedule(d, *t).items()}
        rep = dc.eval_timeline(d, *t, ref["bits"][:, :max(W, 1)].contiguous())
        s = dc.Scheduler(B, L)
        o, got = s.out[d], torch.empty(B, dtype=torch.int64, device="cuda")
        assert dc.dc_schedule_replay_batch(d, B, L, *t, o["makespan"], o["bits"], o["nseg"],
                                           o["status"], got, s.workspace, s.ws_bytes) == dc.DC_OK
        for k in ("makespan", "nseg", "status"):
            assert torch.equal(o[k], ref[k]), (L, d, k)
        if W:
            assert torch.equal(o["bits"], ref["bits"]), (L, d)
        assert torch.equal(got, rep), (L, d)
        n = len(dt) // copies
        bits = ref["bits"][:n, :W].cpu().numpy().view(np.uint32)
        exp = oracle.replay_batch(d, comp[:n], xfer[:n], dt[:n], np.ascontiguousarray(bits),
                                  nthreads=os.cpu_count() or 1)
        assert np.array_equal(got[:n].cpu().numpy(), exp), (L, d)
    assert dc.dc_schedule_replay_batch(2, B, L, *t, None, None, None, None, None, None, 0) == \
        dc.DC_ERR_BAD_SHAPE
    assert dc.dc_schedule_replay_batch(0, B, L, *t, o["makespan"], o["bits"], None, None, None,
                                       s.workspace, s.ws_bytes) == dc.DC_ERR_NULL
