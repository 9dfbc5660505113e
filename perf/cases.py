"""Performance cases: what a program that schedules DynaComm iterations asks of
this library, through the binding's public entry points.

Operations (``op``):

* ``schedule``  forward and backward optimum of profiles resident on the GPU
  (``Scheduler.run``), the library's core call;
* ``step``      one whole step replayed from a CUDA graph (``StepGraph``):
  profile generation, both solves, the timeline replay of both decisions;
* ``fused``     generate and solve without storing the profiles
  (``GeneratedScheduler``);
* ``compare``   the competing strategies on the same profiles: greedy schedulers
  (``greedy``) and layer by layer (``eval_timeline`` of every break), both
  directions;
* ``host``      profiles in pinned host memory, results back on the host
  (``HostPipeline``).

Profiles: the shape tables and device/link draws of ``workloads.config`` for
alexnet (L = 8), vgg16 (16) and resnet50 (54); ``uniform`` layers are the tiny
configuration's draws and ``loguniform`` layers the deep chain's, at any L. Every
result is an integer, so every tolerance is exact.
"""
import math

import numpy as np
import torch

from paper_2101_07968_gb300 import dynacomm as dc
from paper_2101_07968_gb300 import workloads as wl

CNN = {"alexnet": 8, "vgg16": 16, "resnet50": 54}
DIRS = ((0, "fc", "pt"), (1, "bc", "gt"))


def _case(name, op, profile, L, batch):
    return {"name": name, "op": op, "profile": profile, "L": L, "batch": batch}


def listed():
    return [
        # one device asks for its own next iteration, inside the idle window: latency
        _case("one_vgg16", "schedule", "vgg16", 16, 1),
        _case("one_resnet50", "schedule", "resnet50", 54, 1),
        # a small fleet, the whole step as one graph launch: launches and gaps
        _case("tiny_step_4k", "step", "uniform", 8, 4096),
        # a million devices with a shallow model: the shortest rows, bound by memory
        _case("alexnet_1m", "schedule", "alexnet", 8, 1_000_000),
        # the benchmark's own step: a million VGG-16 instances generated, solved, replayed
        _case("vgg16_step_1m", "step", "vgg16", 16, 1_000_000),
        # the same batch without storing its profiles
        _case("vgg16_fused_1m", "fused", "vgg16", 16, 1_000_000),
        # an ordinary deep CNN over a large fleet
        _case("resnet50_262k", "schedule", "resnet50", 54, 262_144),
        # depth sweep: odd depth, ragged batch, long optima
        _case("sweep_l129_20k", "schedule", "loguniform", 129, 20_011),
        # depth sweep: a few hundred very deep, odd-length instances
        _case("sweep_l1023_383", "schedule", "loguniform", 1023, 383),
        # the deepest and largest batch of the configurations
        _case("deepchain_16k", "schedule", "loguniform", 1024, 16_384),
        # strategies compared on one fleet, as in the paper's evaluation
        _case("compare_resnet50_65k", "compare", "resnet50", 54, 65_537),
        # profiles measured on the host, decisions wanted on the host
        _case("host_vgg16_262k", "host", "vgg16", 16, 262_144),
    ]


def draw(rng):
    """A case of the same ranges: batches from one instance to a million, depths
    from 1 to 2048, both spread over their logarithm."""
    op = rng.choice(["schedule"] * 5 + ["step", "fused", "compare", "host"])
    top_l = {"schedule": 2048, "step": 64, "fused": 16, "compare": 200, "host": 64}[op]
    profile = rng.choice(["cnn", "uniform", "loguniform"])
    if profile == "cnn":
        profile = rng.choice([p for p in CNN if CNN[p] <= top_l])
        L = CNN[profile]
    else:
        L = int(round(math.exp(rng.uniform(0.0, math.log(top_l)))))
    elements = {"schedule": 16e6, "step": 16e6, "fused": 16e6, "compare": 3.5e6, "host": 4.2e6}[op]
    cells = {"compare": 2e8}.get(op, 8e11)  # keeps a drawn case below the largest listed one
    power = 2 if op == "compare" else 3
    most = max(1, int(min(1_000_000, elements / L, cells / L ** power)))
    batch = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    return {"op": op, "profile": profile, "L": L, "batch": max(1, batch)}


def _config(case, seed):
    if case["profile"] in CNN:
        cfg = wl.config(case["profile"])
    else:
        cfg = wl.config("tiny" if case["profile"] == "uniform" else "deepchain")
        cfg["L"] = case["L"]
    cfg = wl.with_batch(cfg, case["batch"])
    cfg["seed"] = int(seed)
    return cfg


def prepare(case, seed):
    cfg = _config(case, seed)
    B, L, op = case["batch"], case["L"], case["op"]
    state = {"op": op, "L": L, "batch": B}
    if op == "step":
        state["graph"] = dc.StepGraph(cfg)
    elif op == "fused":
        state["gen"] = dc.GeneratedScheduler(cfg)
    else:
        prof = dc.profile_gen(cfg)
        state["prof"] = prof
        if op == "schedule":
            state["sched"] = dc.Scheduler(B, L)
        elif op == "compare":  # layer by layer: a break after every layer
            words = np.zeros((max(dc.words(L), 1),), dtype=np.uint32)
            for bit in range(L - 1):
                words[bit // 32] |= np.uint32(1 << (bit % 32))
            row = torch.from_numpy(words.view(np.int32)).cuda()
            state["lbl"] = row.expand(B, row.numel()).contiguous()
        elif op == "host":
            host = {k: v.cpu().pin_memory() for k, v in prof.items() if k != "gt"}
            host["gt"] = host["pt"]  # a push moves what its pull moved: one buffer for both
            state["prof"], state["host_in"] = None, host
            state["pipe"] = dc.HostPipeline(B, L)
            state["host_out"] = state["pipe"].host_buffers()
    torch.cuda.synchronize()
    return state


def _outputs(L, out):
    # one layer has no decision word; its placeholder column holds nothing
    return {k: v for k, v in out.items() if L > 1 or k != "bits"}


def run(state):
    op, L, p = state["op"], state["L"], state.get("prof")
    if op == "schedule":
        s = state["sched"]
        return [_outputs(L, s.run(d, p[c], p[x], p["dt"])) for d, c, x in DIRS]
    if op == "step":
        g = state["graph"]
        g.replay()
        return [g.prof] + [dict(_outputs(L, g.sched.out[d]), replay=g.replay_out[d])
                           for d, _, _ in DIRS]
    if op == "fused":
        return _outputs(L, state["gen"].run())
    if op == "compare":
        out = []
        for d, c, x in DIRS:
            out.append(_outputs(L, dc.greedy(d, p[c], p[x], p["dt"])))
            out.append(dc.eval_timeline(d, p[c], p[x], p["dt"], state["lbl"]))
        return out
    state["pipe"].run(state["host_in"], state["host_out"])
    torch.cuda.current_stream().synchronize()  # the results are read on the host
    return [_outputs(L, {k: state["host_out"][(d, k)]
                         for k in ("makespan", "bits", "nseg", "replay")}) for d, _, _ in DIRS]


def work(case):
    """Bytes of one pass: inputs read once, outputs written once. Flops: the two
    prefix additions per layer and direction, which every method needs."""
    B, L, op = case["batch"], case["L"], case["op"]
    W = dc.words(L)
    profile, solved = 8 * (4 * L + 1), 2 * (8 + 4 * W + 4 + 4)
    per = {"schedule": profile + solved,
           "step": profile + solved + 2 * 8,
           "fused": solved,
           "compare": profile + 4 * W + 2 * (8 + 4 * W) + 2 * 8,
           "host": 8 * (3 * L + 1) + 2 * (8 + 4 * W + 4) + 2 * 8}[op]
    return {"bytes": B * per, "flops": 4 * B * L}


def tolerance(case):
    return "exact"


# ------------------------------------------------------------- plain 64 bits
# What `run` returns, in plain torch int64: the generator from its definition, the
# two recurrences cell by cell over every split, the greedy rules by enumeration,
# and the replay layer by layer.
def _i64(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def _shr(z, n):  # logical shift of the 64-bit pattern
    return (z >> n) & ((1 << (64 - n)) - 1)


def _draw64(seed, inst, field, layer):
    z = ((inst << 20) | (field << 12) | layer) + 1
    z = z * _i64(0x9E3779B97F4A7C15) + _i64(seed)
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _uniform(lo, hi, r):
    n = hi - lo + 1
    assert 0 < n < 1 << 31
    return lo + ((_shr(r, 32) * n + (((r & 0xFFFFFFFF) * n) >> 32)) >> 32)


def _loguniform(lo, hi, r):
    knots = [math.floor(lo * math.exp((j / 512) * math.log(hi / lo)) + 0.5) for j in range(513)]
    knots[0], knots[512] = lo, hi
    t = torch.tensor(knots, dtype=torch.int64, device=r.device)
    j, f = _shr(r, 55), _shr(r, 23) & 0xFFFFFFFF
    return t[j] + (((t[j + 1] - t[j]) * f) >> 32)


def _profiles(case, seed):
    cfg = _config(case, seed)
    B, L = case["batch"], case["L"]
    inst = torch.arange(B, dtype=torch.int64, device="cuda")
    one = {}
    for field, key in ((0, "rate"), (1, "bw")):
        dist = _loguniform if cfg[key + "_dist"] == wl.DIST_LOGUNIFORM else _uniform
        one[key] = dist(cfg[key + "_lo"], cfg[key + "_hi"], _draw64(seed, inst, field, 0))[:, None]
    dt = _uniform(cfg["dt_lo"], cfg["dt_hi"], _draw64(seed, inst, 2, 0))
    if cfg["layer_mode"] == wl.LAYERS_FIXED:
        params, flops = (torch.from_numpy(np.asarray(cfg[k], dtype=np.int64)).cuda()[None, :]
                         for k in ("fixed_params", "fixed_flops"))
    else:
        dist = _loguniform if cfg["layer_mode"] == wl.LAYERS_LOGUNIFORM else _uniform
        layer = torch.arange(L, dtype=torch.int64, device="cuda")[None, :]
        params, flops = (dist(cfg[k + "_lo"], cfg[k + "_hi"],
                              _draw64(seed, inst[:, None], field, layer))
                         for field, k in ((3, "params"), (4, "flops")))

    def ceil(a, b):
        return torch.div(a + b - 1, b, rounding_mode="floor")

    pt = ceil(params * (cfg["bits_per_param"] * 1000), one["bw"])
    return {"fc": ceil(flops, one["rate"]), "bc": ceil(flops * cfg["bwd_flops_mult"], one["rate"]),
            "pt": pt, "gt": pt.clone(), "dt": dt}


def _prefix(v):
    return torch.nn.functional.pad(v.cumsum(1), (1, 0))


def _pack(breaks):
    """breaks [B, L+1] bool (position l at column l) -> int32 words [B, max(W, 1)]."""
    B, L = breaks.shape[0], breaks.shape[1] - 1
    out = torch.zeros((B, max(dc.words(L), 1)), dtype=torch.int64, device=breaks.device)
    for l in range(1, L):
        out[:, (l - 1) // 32] |= breaks[:, l].long() << ((l - 1) % 32)
    return torch.where(out >> 31 != 0, out - (1 << 32), out).to(torch.int32)


def _optimum(d, comp, xfer, dt):
    """Eq. 8 / Eq. 9 over every split; ties keep the lowest split and the fewest
    segments."""
    B, L = comp.shape
    if d == 1:
        comp, xfer = comp.flip(1), xfer.flip(1)
    C, X = _prefix(comp), _prefix(xfer)
    S, inf = (C, X)[d], 1 << 60
    late = torch.arange(L + 1, device=comp.device)
    upper = late[None, :, None] > late[None, None, :]  # m > k
    F = torch.full((L + 1, B, L + 1), inf, dtype=torch.int64, device=comp.device)
    dtc = dt[:, None]

    def ready(n):
        return n * dtc + X if d == 0 else C

    tail = S if d == 0 else S + dtc
    F[1, :, 1:] = (ready(1) + tail)[:, 1:]
    for n in range(2, L + 1):
        cand = torch.maximum(F[n - 1][:, None, n - 1:L], ready(n)[:, n:, None]) - S[:, None, n - 1:L]
        cand = torch.where(upper[:, n:, n - 1:L], cand, inf)
        F[n, :, n:] = cand.amin(2) + tail[:, n:]
    T = F[1:, :, L].amin(0)
    order = torch.arange(1, L + 1, device=comp.device)[:, None]
    s = torch.where(F[1:, :, L] == T, order, L + 1).amin(0)
    breaks = torch.zeros((B, L + 1), dtype=torch.bool, device=comp.device)
    rows = torch.arange(B, device=comp.device)
    m = torch.full_like(s, L)
    for n in range(int(s.max()), 1, -1):
        on = s >= n
        cell = F[n, rows, m]
        r = ready(n)[rows, m] if d == 0 else C[rows, m]
        cand = torch.maximum(F[n - 1], r[:, None]) - S + tail[rows, m][:, None]
        hit = (cand == cell[:, None]) & (late[None, :] < m[:, None]) & (F[n - 1] < inf)
        k = torch.where(hit, late[None, :], L + 1).amin(1)
        m = torch.where(on, k, m)
        breaks[rows[on], m[on]] = True
    return T, breaks, s.to(torch.int32)


def _replay(d, comp, xfer, dt, breaks):
    """f_m of a decision, in processing order layer by layer."""
    B, L = comp.shape
    if d == 1:
        comp, xfer = comp.flip(1), xfer.flip(1)
    C, X = _prefix(comp), _prefix(xfer)
    start = torch.zeros(B, dtype=torch.int64, device=comp.device)  # open segment's first prefix
    link, end = torch.zeros_like(dt), torch.zeros_like(dt)
    rows = torch.arange(B, device=comp.device)
    for l in range(1, L + 1):
        close = breaks[:, l] if l < L else torch.ones_like(breaks[:, 0])
        moved, done = X[:, l] - X[rows, start], C[:, l] - C[rows, start]
        if d == 0:
            nl = link + dt + moved
            ne = torch.maximum(end, nl) + done
        else:
            nl = torch.maximum(link, C[:, l]) + dt + moved
            ne = nl
        link, end = torch.where(close, nl, link), torch.where(close, ne, end)
        start = torch.where(close, torch.full_like(start, l), start)
    return end


def _pick(slack, ok):
    """Greedy rule along the last axis: the least non-negative slack, else the
    largest; the first on ties."""
    big = 1 << 60
    good = ok & (slack >= 0)
    least = torch.where(good, slack, big)
    most = torch.where(ok, slack, -big)
    return torch.where(good.any(-1), _first(least == least.amin(-1, keepdim=True)),
                       _first(most == most.amax(-1, keepdim=True)))


def _first(mask):
    idx = torch.arange(mask.shape[-1], device=mask.device)
    return torch.where(mask, idx, mask.shape[-1]).amin(-1)


def _greedy_forward(fc, pt, dt):
    B, L = fc.shape
    breaks = torch.zeros((B, L + 1), dtype=torch.bool, device=fc.device)
    if L < 2:
        return breaks
    C, X = _prefix(fc), _prefix(pt)
    rows, at = torch.arange(B, device=fc.device), torch.arange(L + 1, device=fc.device)
    big = 1 << 60
    a0, b0 = torch.zeros_like(dt), torch.zeros_like(dt)
    have = torch.zeros(B, dtype=torch.bool, device=fc.device)
    wa, wb = torch.ones_like(dt), torch.full_like(dt, 2)
    ws = torch.full_like(dt, -big)
    best = torch.zeros_like(dt)
    for a in range(1, L):
        s = dt[:, None] + X - X[:, a:a + 1] - C[:, a:a + 1]
        s = torch.where(at[None, :] > a, s, -big)
        top = s.amax(1)
        better = top > ws
        ws = torch.where(better, top, ws)
        wa = torch.where(better, torch.full_like(wa, a), wa)
        wb = torch.where(better, _first(s == top[:, None]), wb)
        g = torch.where(s >= 0, s, big)
        low = g.amin(1)
        ok = low < big
        ca, xa = C[rows, a0], X[rows, a0]
        nc, nx = C[:, a], X[:, a]
        better = ok & (~have | (nc > ca) | ((nc == ca) & ((nx < xa) | ((nx == xa) & (low < best)))))
        a0 = torch.where(better, torch.full_like(a0, a), a0)
        b0 = torch.where(better, _first(g == low[:, None]), b0)
        best = torch.where(better, low, best)
        have |= ok
    n, m = torch.where(have, a0, wa), torch.where(have, b0, wb)
    breaks[rows, n] = True
    breaks[rows, m] = True
    while bool((m < L).any()):
        on = m < L
        s = (dt - X[rows, m] - C[rows, m] + C[rows, n])[:, None] + X
        x = _pick(s, at[None, :] > m[:, None])
        n, m = torch.where(on, m, n), torch.where(on, x, m)
        breaks[rows, m] = True
    breaks[:, L] = False
    return breaks


def _greedy_backward(bc, gt, dt):
    B, L = bc.shape
    keep = torch.zeros((B, L + 1), dtype=torch.bool, device=bc.device)
    if L < 2:
        return keep, _replay(1, bc, gt, dt, keep)
    C, X = _prefix(bc), _prefix(gt)
    rows, at = torch.arange(B, device=bc.device), torch.arange(L + 1, device=bc.device)
    least = None
    for q in range(2, L + 1):
        breaks = torch.zeros_like(keep)
        breaks[:, L + 1 - q] = True
        m = torch.full_like(dt, q)
        step = 1
        while bool((m > 1).any()):
            on = m > 1
            s = (step * dt + X[:, L] - X[rows, m - 1] - C[rows, m - 1])[:, None] + C
            x = _pick(s, at[None, :] < (m - 1)[:, None]) + 1  # slack of x sits at x-1
            m = torch.where(on, x, m)
            breaks[rows, L + 1 - m] = True
            step += 1
        breaks[:, L] = False
        t = _replay(1, bc, gt, dt, breaks)
        better = torch.ones_like(on) if least is None else t < least
        least = torch.where(better, t, t if least is None else least)
        keep = torch.where(better[:, None], breaks, keep)
    return keep, least


def _in_pieces(fn, rows, *arrays):
    parts = [fn(*(a[i:i + rows] for a in arrays)) for i in range(0, len(arrays[0]), rows)]
    return [torch.cat(p) for p in zip(*parts)]


def exact(case, seed):
    B, L, op = case["batch"], case["L"], case["op"]
    if B * float(L) ** 3 > 6e11 or (op == "compare" and B * float(L) ** 3 > 2e11):
        return None
    p = _profiles(case, seed)
    rows = max(1, int(4e7 / (L + 1) ** 2))
    out, fused = [], {"makespan": [], "bits": [], "nseg": [], "status": []}
    if op == "step":
        out.append(p)
    for d, c, x in DIRS:
        if op == "compare":
            if d == 0:
                breaks, = _in_pieces(lambda *a: (_greedy_forward(*a),), rows, p[c], p[x], p["dt"])
                span = _replay(0, p[c], p[x], p["dt"], breaks)
            else:
                breaks, span = _in_pieces(_greedy_backward, rows, p[c], p[x], p["dt"])
            out.append(_outputs(L, {"makespan": span, "bits": _pack(breaks)}))
            out.append(_replay(d, p[c], p[x], p["dt"], torch.ones_like(breaks)))
            continue
        T, breaks, s = _in_pieces(lambda *a, d=d: _optimum(d, *a), rows, p[c], p[x], p["dt"])
        one = {"makespan": T, "bits": _pack(breaks), "nseg": s, "status": torch.zeros_like(s)}
        for k in fused:
            fused[k].append(one[k])
        if op in ("step", "host"):
            one["replay"] = _replay(d, p[c], p[x], p["dt"], breaks)
        if op == "host":
            del one["status"]
        out.append(_outputs(L, one))
    if op == "fused":
        return _outputs(L, {k: torch.stack(v) for k, v in fused.items()})
    return out
