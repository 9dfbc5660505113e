"""dc_step_batch (StepGraph's one-pass step) against the separate calls: profiles,
decisions and replays bit for bit, for odd and even depths, ragged tiles, both division
forms, listed instances and unaligned profile arrays."""
import pytest

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


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("name,L,batch,kw", [
    ("vgg16", 16, 70_003, {}), ("alexnet", 8, 65_537, {}), ("deepchain", 11, 65_600, {}), ("tiny", 8, 33, {}),
    ("deepchain", 1, 100, {}), ("deepchain", 2, 70, {}), ("deepchain", 5, 999, {}),
    ("deepchain", 11, 3001, {}), ("deepchain", 12, 3001, {}), ("deepchain", 15, 40_001, {}),
    ("vgg16", 16, 5000, dict(bw_lo=1, bw_hi=50, dt_hi=2**33)), ("alexnet", 8, 1, {}),
    ("tiny", 8, 7999, {}), ("tiny", 8, 8001, {}), ("tiny", 16, 8000, {}), ("deepchain", 16, 6000, {}),
    ("deepchain", 16, 6001, {}), ("deepchain", 7, 2, {}), ("tiny", 3, 4097, dict(bw_hi=2000, dt_hi=2**40)),
    ("vgg16", 16, 9001, dict(bw_lo=1, bw_hi=50, dt_hi=2**33))])
def test_one_pass_step(dc, name, L, batch, kw, offset):
    import torch
    cfg = wl.with_batch(wl.config(name), batch, inst0=7)
    cfg.update(L=L, **kw)
    ref = dc.profile_gen(cfg)

    def buf(*shape, dtype=torch.int64):  # offset 1: 8 bytes past a 16-byte boundary
        n = 1
        for s in shape:
            n *= s
        return torch.empty(n + offset, dtype=dtype, device="cuda")[offset:].view(*shape)

    p = {k: buf(batch, L) for k in ("fc", "pt", "bc", "gt")}
    p["dt"] = buf(batch)
    W = dc.words(L)
    o = {"makespan": buf(2, batch), "replay": buf(2, batch),
         "bits": torch.zeros((2, batch, max(W, 1)), dtype=torch.int32, device="cuda"),
         "nseg": torch.empty((2, batch), dtype=torch.int32, device="cuda"),
         "status": torch.empty((2, batch), dtype=torch.int32, device="cuda")}
    n = dc.dc_schedule_generated_workspace_bytes(batch, L)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    args = (o["makespan"], o["bits"], o["nseg"], o["status"], o["replay"], ws)
    assert dc.dc_step_batch(cfg, p["fc"], p["pt"], p["bc"], p["gt"], p["dt"], *args, n) == dc.DC_OK
    for k in p:
        assert torch.equal(p[k], ref[k]), k
    for d, (c, x) in ((0, ("fc", "pt")), (1, ("bc", "gt"))):
        exp = dc.schedule(d, ref[c], ref[x], ref["dt"])
        for k in ("makespan", "nseg", "status") + (("bits",) if W else ()):
            assert torch.equal(o[k][d], exp[k]), (k, d)
        rep = dc.eval_timeline(d, ref[c], ref[x], ref["dt"], exp["bits"])
        assert torch.equal(o["replay"][d], rep), d
    if dc.fused_step(batch, L, cfg["layer_mode"]) and not offset:
        g = dc.StepGraph(cfg)
        for _ in range(2):
            g.replay()
        torch.cuda.synchronize()
        for d in (0, 1):
            assert torch.equal(g.sched.out[d]["makespan"], o["makespan"][d])
            assert torch.equal(g.replay_out[d], o["replay"][d])
            assert torch.equal(g.prof["bc"], ref["bc"])


def test_arguments(dc):
    import torch
    cfg = wl.with_batch(wl.config("alexnet"), 10)
    b = torch.empty(10_000, dtype=torch.int64, device="cuda")
    n = dc.dc_schedule_generated_workspace_bytes(10, 8)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    ok = [b, b, b, b, b, b, b, None, None, b, ws]
    for miss in (0, 4, 5, 6, 9):
        bad = list(ok)
        bad[miss] = None
        assert dc.dc_step_batch(cfg, *bad, n) == dc.DC_ERR_NULL, miss
    assert dc.dc_step_batch(cfg, *ok, n - 1) == dc.DC_ERR_WORKSPACE
    deep = wl.with_batch(wl.config("resnet50"), 10)
    assert dc.dc_step_batch(deep, *ok, n) == dc.DC_ERR_BAD_SHAPE
