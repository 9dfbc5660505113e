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
