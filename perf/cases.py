"""Timed cases of the load anticipator and the load-aware router, through `DeviceState`.

One pass is one cycle of a serving control loop on one GPU: the maps are built from the serving engine's request table
(`anticipate`), then come `ticks` scheduler ticks, each a decode iteration (`decode`: `step`, or `tick` with the
refinement against real lengths and the scaler's signals) followed by the routing of the tick's arrivals.  The engine's
columns that a pass changes are put back from its copy at the start, as a loop that takes its table from the engine does,
so every pass of a state does the same work.

Sizes are those of the five seeded configurations (`workloads.make_config`, 0 to 4) or generic; lengths are log-normal
with the medians, spreads and clamps of configurations 0-1 ("chat") and 2-4 ("long"), tokens generated uniform below the
predicted length.  The capacity puts the median instance's present occupancy at the share `load` of the capacity (0.8 is
the router's ideal usage: the penalty term decides routes for about half of the instances).

Fields of a case
  instances, horizon, requests   I, H and in-flight requests
  arrivals, ticks                arrivals per tick and ticks per pass (0 ticks: the build alone)
  lengths, zipf                  length distributions; instances drawn by Zipf(1.1) instead of uniformly
  decode, refine, signals        the decode iteration and what rides on it
  width                          full-width maps of that many steps kept as a ring, `horizon` being the window (0: dense maps)
  queue                          room of the admission queue (0: plain router)
  load, whole, beta              capacity; whether t_mem * M is a whole number (a KV cache of 16-token blocks seldom gives
                                 one); penalty coefficient of the router
"""
from __future__ import annotations

import math

import torch

from paper_2504_03702_b200 import binding as B
from paper_2504_03702_b200.state import DeviceState

DEVICE = "cuda:0"
T_MEM = 0.8
# (prompt median, sigma, lo, hi), (output median, sigma, lo, hi)
LENGTHS = {
    "chat": ((512, 1.0, 16, 4096), (256, 1.0, 1, 2048)),
    "long": ((1024, 1.2, 16, 8192), (384, 1.2, 1, 4096)),
}


def _case(**kw):
    c = dict(instances=64, horizon=256, requests=16384, arrivals=0, ticks=1, lengths="long", zipf=False, decode=True,
             refine=False, signals=False, width=0, queue=0, load=0.8, whole=True, beta=1.0)
    c.update(kw)
    return c


def listed():
    return [
        # one request routed on freshly built maps of a small service: the latency a request waits for
        _case(name="route_one", instances=8, horizon=64, requests=256, arrivals=1, lengths="chat", decode=False),
        # configuration 0: one tick of a small service
        _case(name="tiny", instances=8, horizon=64, requests=256, arrivals=32, lengths="chat"),
        # configuration 1
        _case(name="small", instances=64, horizon=256, requests=16384, arrivals=1024, lengths="chat"),
        # configuration 2: skewed load, one instance holds a seventh of the requests
        _case(name="medium_zipf", instances=512, horizon=1024, requests=262144, arrivals=8192, zipf=True),
        # configuration 3: the largest one-shot batch, the headline workload of the benchmark
        _case(name="large", instances=4096, horizon=2048, requests=2097152, arrivals=65536),
        # configuration 4: four ticks of the stream with everything a tick can carry
        _case(name="stream", instances=1024, horizon=1024, requests=524288, arrivals=4096, ticks=4, refine=True,
              signals=True),
        # the anticipator alone on the largest configuration (a service that rebuilds its maps from the engine)
        _case(name="build_large", instances=4096, horizon=2048, requests=2097152, ticks=0),
        # decode ticks without arrivals on the largest configuration
        _case(name="tick_large", instances=4096, horizon=2048, requests=2097152, ticks=8, refine=True, signals=True),
        # full-width maps with the paper's widths (L = 4,096, l = 100)
        _case(name="ring", instances=256, horizon=100, width=4096, requests=65536, arrivals=1024, ticks=4, refine=True),
        # admission queue of a service close to its limit
        _case(name="admit", instances=512, horizon=1024, requests=131072, arrivals=2048, ticks=4, queue=1024, load=0.97,
              signals=True),
        # odd sizes, a penalty coefficient below one: binary64 scores
        _case(name="ragged", instances=333, horizon=777, requests=70001, arrivals=1501, ticks=2, whole=False, beta=0.75,
              lengths="chat", refine=True),
        # a larger service whose capacity is a number of 16-token blocks: binary64 scores with beta = 1
        _case(name="blocks", instances=2000, horizon=1536, requests=600000, arrivals=8192, whole=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    inst = _log(rng, 4, 4096)
    horizon = _log(rng, 40, 2048)
    per = _log(rng, 32, 512)
    requests = min(inst * per + rng.randrange(inst), 2000000)
    kind = rng.choice(("batch", "batch", "batch", "ticks", "ticks", "admit", "ring", "build"))
    whole = rng.random() < 0.6
    c = _case(instances=inst, horizon=horizon, requests=requests, lengths=rng.choice(("chat", "long")),
              zipf=rng.random() < 0.25, whole=whole, beta=1.0 if whole or rng.random() < 0.5 else 0.75)
    if kind == "build":
        c["ticks"] = 0
        return c
    c["arrivals"] = _log(rng, 1, 8192)
    if kind == "batch":
        c["decode"] = rng.random() < 0.7
        return c
    c["ticks"] = rng.randrange(1, 5)
    c["arrivals"] = max(1, c["arrivals"] // c["ticks"])
    c["refine"] = rng.random() < 0.5
    if kind == "ring":
        c["horizon"] = _log(rng, 64, 256)
        c["width"] = _log(rng, 1024, 4096)
        c["instances"] = min(c["instances"], 2048)
        c["requests"] = min(c["requests"], c["instances"] * per)
    elif kind == "admit":
        c["queue"] = _log(rng, 16, 2048)
        c["load"] = rng.choice((0.8, 0.97, 1.6))
        c["signals"] = rng.random() < 0.5
    else:
        c["signals"] = rng.random() < 0.5
    return c


def _lognormal(gen, n, spec):
    median, sigma, lo, hi = spec
    z = torch.randn(n, generator=gen, device=DEVICE, dtype=torch.float64)
    return torch.exp(math.log(median) + sigma * z).round().clamp(lo, hi).to(torch.int32)


def _instances(gen, n, inst, zipf):
    u = torch.rand(n, generator=gen, device=DEVICE, dtype=torch.float64)
    if not zipf:
        return (u * inst).to(torch.int32).clamp(max=inst - 1)
    w = torch.arange(1, inst + 1, device=DEVICE, dtype=torch.float64) ** -1.1
    cdf = torch.cumsum(w, 0)
    return torch.searchsorted(cdf / cdf[-1], u, right=True).clamp(max=inst - 1).to(torch.int32)


def _actual(gen, predicted, generated):
    """Real response lengths: the prediction plus a two-component Laplace error (mean absolute error 78 tokens)."""
    n = predicted.shape[0]
    near = torch.rand(n, generator=gen, device=DEVICE, dtype=torch.float64) < 0.7
    u = torch.rand(n, generator=gen, device=DEVICE, dtype=torch.float64) - 0.5
    scale = torch.where(near, 20.0, 214.17)
    err = -scale * torch.sign(u) * torch.log1p(-2.0 * u.abs().clamp(max=0.4999999))
    act = (predicted.double() + err).round().to(torch.int32)
    return torch.maximum(act, generated + 1).clamp(min=1)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    inst, n = case["instances"], case["requests"]
    a, ticks = case["arrivals"], case["ticks"]
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    p_spec, d_spec = LENGTHS[case["lengths"]]
    prompt = _lognormal(gen, n, p_spec)
    predicted = _lognormal(gen, n, d_spec)
    u = torch.rand(n, generator=gen, device=DEVICE, dtype=torch.float64)
    generated = torch.minimum((u * predicted).to(torch.int32), predicted - 1)
    instance = _instances(gen, n, inst, case["zipf"])
    s.arrivals = [(_lognormal(gen, a, p_spec), _lognormal(gen, a, d_spec)) for _ in range(ticks if a else 0)]
    # capacity: the median instance's tokens are the share `load` of it
    held = torch.zeros(inst, dtype=torch.int64, device=DEVICE)
    held.scatter_add_(0, instance.long(), (prompt + generated).long())
    median = max(int(held.median()), 1)
    m = 5 * max(1, round(median / case["load"] / 5))
    if not case["whole"]:   # a number of 16-token blocks that is no multiple of five
        blocks = max(1, m // 16)
        m = 16 * (blocks + 1 if blocks % 5 == 0 else blocks)
    total = n + (a * ticks)
    st = DeviceState(inst, case["horizon"], m, total, T_MEM, case["beta"], device=DEVICE)
    st.load_requests(prompt.cpu().numpy(), generated.cpu().numpy(), predicted.cpu().numpy(), instance.cpu().numpy())
    s.st = st
    s.n0 = torch.tensor([n], dtype=torch.int64, device=DEVICE)
    s.generated0, s.predicted0 = generated, predicted
    s.actual = None
    if case["refine"]:
        tail_d = [d for _, d in s.arrivals]
        d = torch.cat([predicted] + tail_d)
        g = torch.cat([generated, torch.zeros(total - n, dtype=torch.int32, device=DEVICE)])
        s.actual = _actual(gen, d, g)
    if case["queue"]:
        st.make_queue(case["queue"])
    s.builder = None
    if case["width"]:
        code, s.builder = B.pre_create(inst, case["width"], m, T_MEM, case["beta"], total)
        B.check(code, "pre_create")
        st.make_ring(case["width"], builder=s.builder)
    return s


def run(s):
    c, st = s.case, s.st
    n = c["requests"]
    out = {}
    # ---- the table as the engine has it
    if c["decode"] and c["ticks"]:
        st.generated[:n].copy_(s.generated0)
        if c["refine"]:
            st.predicted[:n].copy_(s.predicted0)
    if c["ticks"]:
        st.n_requests.copy_(s.n0)
        st.queued_p.zero_()
    if c["queue"]:
        st.queue_state.zero_()
    # ---- the maps
    if c["width"]:
        st.head.zero_()
        B.check(B.pre_anticipate(s.builder, st.prompt, st.generated, st.predicted, st.instance, n, st.ring,
                                 st.current_d), "pre_anticipate")
    else:
        st.anticipate(n)
    # ---- the ticks
    for t in range(c["ticks"]):
        if c["width"]:
            if c["decode"]:
                st.ring_step()
                if c["refine"]:
                    out["counts%d" % t] = st.ring_refine(s.actual)
            st.ring_window()
        elif c["decode"]:
            if c["refine"] or c["signals"]:
                counts, over, row_max, summary = st.tick(s.actual, c["signals"])
                if c["refine"]:
                    out["counts%d" % t] = counts
                if c["signals"]:
                    out["signals%d" % t] = (over, row_max, summary)
            else:
                st.step()
        if c["arrivals"]:
            p, d = s.arrivals[t]
            if c["queue"]:
                waited, choice, score = st.route_admit(p, d)
                out["routes%d" % t] = (choice, score)
                out["waited"] = waited
                out["queue"] = st.queue_state
            else:
                choice, score = st.route_batch(p, d)
                out["routes%d" % t] = (choice, score)
            if c["width"]:
                st.ring_fold(p, d, choice)
    out["maps"] = st.ring if c["width"] else st.curves
    out["current_d"] = st.current_d
    if c["ticks"]:
        out["table"] = (st.prompt, st.generated, st.predicted, st.instance, st.n_requests)
        out["queued_p"] = st.queued_p
    return out


def _mean(spec, top):
    """Mean of a clamped log-normal cut at `top`, by the midpoint rule over its quantiles."""
    median, sigma, lo, hi = spec
    total, k = 0.0, 200
    for i in range(k):
        q = (i + 0.5) / k
        z = math.sqrt(2.0) * _erfinv(2.0 * q - 1.0)
        total += min(max(median * math.exp(sigma * z), lo), min(hi, top))
    return total / k


def _erfinv(y):
    x = 0.0
    lo, hi = -6.0, 6.0
    for _ in range(60):
        x = 0.5 * (lo + hi)
        if math.erf(x) < y:
            lo = x
        else:
            hi = x
    return x


def work(case):
    """Each call's inputs once and its outputs once.  Operations: the score of every arrival against every instance (three
    each) and one addition per map cell that a request reaches."""
    inst, n, a, ticks = case["instances"], case["requests"], case["arrivals"], case["ticks"]
    width = case["width"] or case["horizon"]
    d_spec = LENGTHS[case["lengths"]][1]
    reach = _mean(d_spec, width)
    cells = 8.0 * inst * width
    window = 8.0 * inst * case["horizon"]
    total = 16.0 * n + cells + 8.0 * inst                      # the build
    ops = n * 2.0 + inst * width * 2.0
    for t in range(ticks):
        rows = n + a * t
        if case["decode"]:
            total += 20.0 * rows + (4.0 * rows if case["refine"] else 0.0) + 32.0 * inst
            total += 16.0 * inst if case["width"] else 2.0 * cells
            if case["signals"]:
                total += 12.0 * inst
        if case["width"]:
            total += 2.0 * window
        if a:
            total += window + 16.0 * inst + 36.0 * a
            total += 16.0 * min(a * reach, inst * width) + 32.0 * min(a, inst)
            ops += 3.0 * a * inst + a * reach
    return {"bytes": total, "flops": ops}


def tolerance(case):
    """Whole numbers (maps, routes, table) and scores whose operations are fixed one by one: the same bits."""
    return "exact"
