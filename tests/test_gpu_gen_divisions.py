"""The generator's two divisions: quotients below 2^32 in 32-bit steps, any other config
in 64-bit ones. Configs on both sides of the line and at the ends of the divisors' range,
in every batch size that changes the kernel's tiles, every value equal to the oracle's;
generate-and-solve equal to the separate calls."""
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


def _cfg(name, batch, **kw):
    cfg = wl.with_batch(wl.config(name), batch, inst0=kw.pop("inst0", 0))
    if name == "deepchain":
        cfg["L"] = kw.pop("L", 13)
    cfg.update(kw)
    return cfg


# the largest VGG-16 layer sends 102,764,544 params * 32,000: a quotient of 2^32 at 765 kbit/s
CASES = [("vgg16", dict(bw_lo=766, bw_hi=4000)), ("vgg16", dict(bw_lo=765, bw_hi=4000)),
         ("vgg16", dict(bw_lo=1, bw_hi=2**31 - 1, rate_lo=1, rate_hi=2**31 - 1)),
         ("vgg16", dict(rate_lo=2**30, rate_hi=2**31 - 1, bw_lo=2**30, bw_hi=2**31 - 1)),
         ("alexnet", dict(bwd_flops_mult=1)), ("alexnet", dict(bwd_flops_mult=3)),
         ("alexnet", dict(bwd_flops_mult=16, bits_per_param=64)),
         ("tiny", dict(rate_lo=1, rate_hi=3)), ("tiny", dict(params_lo=0, flops_lo=0)),
         ("deepchain", dict()), ("deepchain", dict(flops_hi=2**40, params_hi=2**40)),
         ("resnet50", dict(seed=2**63 + 5, inst0=2**43))]


@pytest.mark.parametrize("name,kw", CASES)
@pytest.mark.parametrize("batch", [1, 37, 3000, 50_001])
def test_every_value(dc, name, kw, batch):
    import torch
    cfg = _cfg(name, batch, **dict(kw))
    got = dc.profile_gen(cfg)
    exp = oracle.profile_gen(cfg)
    for k in ("fc", "pt", "bc", "gt", "dt"):
        assert np.array_equal(got[k].cpu().numpy(), exp[k]), k
    if cfg["L"] <= 16 and batch <= 3000:
        out = dc.GeneratedScheduler(cfg).run()
        for d, (c, x) in ((0, ("fc", "pt")), (1, ("bc", "gt"))):
            ref = dc.schedule(d, got[c], got[x], got["dt"])
            for k in ("makespan", "bits", "nseg", "status"):
                assert torch.equal(out[k][d], ref[k]), (k, d)


# Numerators at the 32-bit steps' upper edge, d * 2^32 - 1 and its neighbours: the largest
# cost is the QUOTIENT ROUNDED UP, 2^32 - 1 (in 32 bits) or 2^32 (not in 32 bits).
def _edge(rate, flops, mult=2, bits=32, params=(1, 2, 3, 4), bw=1000):
    cfg = wl.config("vgg16")
    cfg.update(L=len(flops), fixed_flops=list(flops), fixed_params=list(params),
               rate_lo=rate, rate_hi=rate, bw_lo=bw, bw_hi=bw, bits_per_param=bits,
               bwd_flops_mult=mult)
    return cfg


K = 2**32
EDGES = [_edge(d, (f, 1, 0, d), mult)
         for d in (2, 3, 255) for mult in (1, 2)
         for f in ((K - 1) * d, (K - 1) * d + 1, K * d - 1, K * d)]
EDGES += [_edge(d, (f, 1, 0, d), 3)
          for d in (2, 3, 255) for f in ((K - 1) * d // 3, (K - 1) * d // 3 + 1, K * d // 3)]
EDGES += [_edge(1000, (1, 2, 3, 4), 2, bits, (p, 1, 0, 2), bw)
          for bits, p, bw in ((32, 35_030_827, 261), (1, 4_299_262_263, 1001),
                              (1, 4_299_262_262, 1001), (1, 4_299_262_264, 1001))]


@pytest.mark.parametrize("edge", range(len(EDGES)))
@pytest.mark.parametrize("batch", [37, 9000, 70_001])  # every generator and generate-and-solve kernel
def test_costs_at_two_to_the_32(dc, edge, batch):
    import torch
    cfg = wl.with_batch(EDGES[edge], batch)
    got = dc.profile_gen(cfg)
    exp = oracle.profile_gen(cfg)
    for k in ("fc", "pt", "bc", "gt", "dt"):
        assert np.array_equal(got[k].cpu().numpy(), exp[k]), k
    ref = {d: dc.schedule(d, got[c], got[x], got["dt"])
           for d, c, x in ((0, "fc", "pt"), (1, "bc", "gt"))}
    out = dc.GeneratedScheduler(cfg).run()
    for d in (0, 1):
        for k in ("makespan", "bits", "nseg", "status"):
            assert torch.equal(out[k][d], ref[d][k]), (k, d)
    g = dc.StepGraph(cfg)
    g.replay()
    torch.cuda.synchronize()
    for k in ("fc", "pt", "bc", "gt", "dt"):
        assert np.array_equal(g.prof[k].cpu().numpy(), exp[k]), k


@pytest.mark.parametrize("batch", [16_000, 16_001, 24_000, 24_001])
@pytest.mark.parametrize("name,L", [("alexnet", 0), ("tiny", 1), ("tiny", 10), ("deepchain", 3), ("deepchain", 17)])
def test_tables_in_shared_memory_or_not(dc, name, L, batch):
    """Both sides of the line between reading the tables from the parameters and copying
    them, and of the number of instances to a tile."""
    cfg = wl.with_batch(wl.config(name), batch, inst0=5)
    cfg["L"] = L or cfg["L"]
    got, exp = dc.profile_gen(cfg), oracle.profile_gen(cfg)
    for k in ("fc", "pt", "bc", "gt", "dt"):
        assert np.array_equal(got[k].cpu().numpy(), exp[k]), k
