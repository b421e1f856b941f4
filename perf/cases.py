"""What the scheduler library is timed on: the calls a serving control plane makes, through the package's own classes.

A case is a dict of plain values; its "kind" says which call or loop of calls it is:

  step      Scheduler.step over a request table: one decision (steps = 0), or a look-ahead of `steps` committed
            iterations from a snapshot that is copied back first
  dispatch  Scheduler.dispatch_step: the global queue handed to the instances that are due
  sim       Scheduler.sim_run: a batch of independent traces
  pd        rounds of the disaggregated loop from a snapshot: committed step, hand-off P -> D
  elastic   rounds of the scaling loop from a snapshot: committed steps under a horizon, Scaler tick and its decisions,
            dispatch, binding
  monitor   attainment of a table, and the SLO targets of newly arrived requests from a window of finished ones

Sizes, SLO classes, latency model and distributions are those of gen/workloads.py, bench.py and the tests; the inputs are drawn on the
GPU from the seed alone.  All results are integers.
"""
import math

import numpy as np
import torch

import gen
import paper_2508_15919_b200 as hfx
from gen import workloads as W

MS, SEC = W.MS, W.SEC
NOW = 1000 * SEC
SLO_BOUNDS = ("ttft_min_ns", "ttft_max_ns", "ttft_min_relaxed_ns", "tpot_min_ns", "tpot_max_ns", "tpot_min_relaxed_ns")
MUTABLE = ("state", "gen", "first_token_ns", "last_token_ns", "finish_ns")


def _step(name, rows, replicas, **kw):
    """A table of `rows` requests on `replicas` instances.  layout: rows grouped by instance, or interleaved in arrival order
    (one shared queue).  inflight / done / future: shares of the rows that are decoding, finished, not arrived yet.
    ids: request ids rise with the rows (one front end numbers them), or not (several do).  outputs: also the optional ones."""
    c = dict(name=name, kind="step", rows=rows, replicas=replicas, stages="colocated", layout="interleaved", lengths="lognormal", classes=4,
             inflight=0.2, done=0.0, future=0.0, ids="rising", weights=False, first_fit=False, cap_only=False, outputs="required", steps=0)
    c.update(kw)
    return c


def listed():
    return [
        # one instance with a short queue, all outputs: what a single server's scheduler asks between two iterations; latency counts
        _step("step 1x256", 256, 1, classes=3, inflight=0.1, future=0.5, outputs="all"),
        # a rack of instances, each with its own rows, most of them decoding; capacity limits only, all outputs
        _step("step 64x4096 grouped", 64 * 4096, 64, layout="grouped", inflight=0.6, cap_only=True, outputs="all"),
        # the largest: disaggregated fleet, deep queues on the prefill side, prefilled requests waiting on the decode side
        _step("step 128P+128D x16384", 256 * 16384, 256, stages="pd", layout="grouped", lengths="bimodal", classes=0),
        # one shared arrival-ordered queue over a large fleet, priority weights: ten committed iterations of look-ahead
        _step("rollout 1M over 1024", 1 << 20, 1024, lengths="pareto", classes=5, inflight=0.1, future=0.5, weights=True, steps=10),
        # a ragged table whose ids do not rise with the rows, old rows not yet cleared, first-fit admission
        _step("step 300007 permuted first fit", 300_007, 96, classes=0, inflight=0.3, done=0.15, future=0.2, ids="permuted", first_fit=True,
              outputs="all"),
        # a planner replays one trace of one instance
        dict(name="sim 1x256", kind="sim", traces=1, rows=256, ragged=False, bursty=False, iterations=2000, first_fit=False),
        # Monte-Carlo capacity planning: thousands of bursty traces
        dict(name="sim 4096x2048", kind="sim", traces=4096, rows=2048, ragged=False, bursty=True, iterations=10000, first_fit=False),
        # the central dispatcher of a large fleet with a deep global queue
        dict(_step("dispatch 1M over 1024", 1 << 20, 1024, lengths="pareto", classes=5, inflight=0.1, future=0.5, weights=True), kind="dispatch"),
        # dispatcher and migrator of a disaggregated fleet, ids from several front ends
        dict(_step("dispatch 60013 16P+16D permuted", 60_013, 32, stages="pd", classes=0, inflight=0.3, done=0.1, future=0.2, ids="permuted"),
             kind="dispatch"),
        # the disaggregated loop in mid-run: ten rounds of committed step and hand-off
        dict(name="pd loop 1M 128+128", kind="pd", rows=1 << 20, replicas=256, ids="rising", rounds=10),
        # the scaling loop in mid-run: four ticks of 50 ms
        dict(name="elastic loop 1M over 1024", kind="elastic", rows=1 << 20, replicas=1024, rounds=4),
        # what a dashboard and the SLO mapper ask once per tick
        dict(name="monitor 1M window 4096", kind="monitor", rows=1 << 20, window=4096, requests=10_000, priorities=4),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["sim"] * 2 + ["dispatch"] * 2 + ["pd", "elastic", "monitor"])
    if kind == "sim":
        rows = _log(rng, 64, 4096)
        traces = _log(rng, 1, min(4096, 4096 * 2048 // rows))
        return dict(kind=kind, traces=traces, rows=rows, ragged=rng.random() < 0.5, bursty=rng.random() < 0.7, iterations=_log(rng, 500, 10000),
                    first_fit=rng.random() < 0.25)
    if kind == "monitor":
        return dict(kind=kind, rows=_log(rng, 1000, 1 << 20), window=_log(rng, 64, 4096), requests=_log(rng, 16, 100_000), priorities=rng.randint(1, 16))
    if kind in ("pd", "elastic"):
        replicas = _log(rng, 4, 1024) & ~1
        rows = _log(rng, max(256, 8 * replicas), 1 << 20)
        if kind == "pd":
            return dict(kind=kind, rows=rows, replicas=replicas, ids=rng.choice(["rising", "permuted"]), rounds=rng.randint(2, 10))
        return dict(kind=kind, rows=rows, replicas=replicas, rounds=rng.randint(1, 4))
    pd = rng.random() < 0.3
    replicas = _log(rng, 2 if pd else 1, 4096 if kind == "dispatch" else 2048)
    steps = rng.randint(1, 10) if kind == "step" and rng.random() < 0.4 else 0
    per = 16384 if not steps else 4096      # rows of one instance
    rows = _log(rng, min(256, replicas * per), min(replicas * per, (1 << 20) if steps or kind == "dispatch" else 1 << 22))
    c = _step("", rows, replicas, stages="pd" if pd else "colocated", layout=rng.choice(["grouped", "interleaved"]),
              lengths=rng.choice(["lognormal", "pareto", "bimodal"]), classes=rng.choice([0, 3, 4, 5]), inflight=round(rng.uniform(0.02, 0.6), 3),
              done=round(rng.uniform(0.0, 0.2), 3), future=round(rng.choice([0.0, rng.uniform(0.1, 0.5)]), 3), ids=rng.choice(["rising", "rising", "permuted"]),
              weights=rng.random() < 0.3, first_fit=rng.random() < 0.2, cap_only=rng.random() < 0.2, outputs=rng.choice(["all", "required"]), steps=steps)
    del c["name"]
    c["kind"] = kind
    if kind == "dispatch":
        c.update(outputs="required", first_fit=False, layout="interleaved")
    return c


# ---- inputs ------------------------------------------------------------------------------------------------
class _Draw:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def u(self, *n):
        return torch.rand(*n, generator=self.g, device="cuda", dtype=torch.float64)

    def ints(self, lo, hi, n):      # lo .. hi - 1
        return torch.randint(lo, hi, (n,), generator=self.g, device="cuda", dtype=torch.int64)

    def exp(self, mean, n):
        return -torch.log1p(-self.u(n)) * mean

    def normal(self, n):
        return torch.randn(n, generator=self.g, device="cuda", dtype=torch.float64)

    def lognormal(self, mu, sigma, lo, hi, n):
        return torch.exp(mu + sigma * self.normal(n)).round().clamp(lo, hi).to(torch.int32)

    def prompts(self, lengths, n, hi=8192):
        if lengths == "pareto":
            return (16.0 * (1.0 - self.u(n)) ** (-1.0 / 1.5)).round().clamp(16, 131072).to(torch.int32)
        if lengths == "bimodal":
            short, long_ = torch.exp(5.0 + 0.7 * self.normal(n)), torch.exp(9.0 + 0.5 * self.normal(n))
            return torch.where(self.u(n) < 0.7, short, long_).round().clamp(16, 131072).to(torch.int32)
        return self.lognormal(6.0, 1.0, 16, hi, n)

    def permutation(self, n):
        return torch.randperm(n, generator=self.g, device="cuda")


def _ns(x):
    return x.round().to(torch.int64)


def _classes(k):
    return {0: W.CLASSES_PD, 3: W.CLASSES_3, 4: W.CLASSES_4, 5: W.CLASSES_5}[k]


def _empty(n):
    dt = {"class_id": torch.uint8, "state": torch.uint8, "arrival_ns": torch.int64, "first_token_ns": torch.int64, "last_token_ns": torch.int64,
          "finish_ns": torch.int64}
    t = {k: torch.zeros(n, dtype=dt.get(k, torch.int32), device="cuda") for k in W._empty_table(1)}
    t["req_id"] = torch.arange(n, dtype=torch.int32, device="cuda")
    t["weight"] += 1
    return t


def _in_flight(d, t, m, classes, now):
    """Rows of the mask m are decoding: gen ~ U[0, output_len), first token gen * tpot * U[0.5, 1.2] ago, arrival before that."""
    n = m.shape[0]
    tpot = torch.tensor([c[1] if c[1] > 0 else 100 * MS for c in classes], device="cuda", dtype=torch.float64)[t["class_id"].long()]
    g = torch.floor(d.u(n) * t["output_len"])
    first = now - _ns(g * tpot * (0.5 + 0.7 * d.u(n))) - _ns(d.u(n) * 20 * MS)
    arrival = first - _ns((0.05 + 0.95 * d.u(n)) * SEC)
    t["state"] = torch.where(m, W.RUNNING, t["state"]).to(torch.uint8)
    t["gen"] = torch.where(m, g.to(torch.int32), t["gen"])
    t["first_token_ns"] = torch.where(m, first, t["first_token_ns"])
    t["last_token_ns"] = torch.where(m, now - _ns(d.u(n) * 20 * MS), t["last_token_ns"])
    t["arrival_ns"] = torch.where(m, torch.minimum(t["arrival_ns"], arrival), t["arrival_ns"])


def _finished(d, t, m, classes, now):
    """Rows of the mask m are finished: about half of them within their targets."""
    n = m.shape[0]
    tpot = torch.tensor([c[1] if c[1] > 0 else 100 * MS for c in classes], device="cuda", dtype=torch.float64)[t["class_id"].long()]
    ttft = torch.tensor([c[0] if c[0] > 0 else 10 * SEC for c in classes], device="cuda", dtype=torch.float64)[t["class_id"].long()]
    first = t["arrival_ns"] + _ns(ttft * d.exp(0.8, n))
    last = first + _ns(tpot * (0.3 + 0.9 * d.u(n)) * (t["output_len"] - 1).clamp(min=0))
    t["state"] = torch.where(m, W.DONE, t["state"]).to(torch.uint8)
    t["gen"] = torch.where(m, (t["output_len"] - 1).clamp(min=0), t["gen"])
    t["first_token_ns"] = torch.where(m, first, t["first_token_ns"])
    for k in ("last_token_ns", "finish_ns"):
        t[k] = torch.where(m, last, t[k])


def _table(case, d):
    """Request table, instance configuration and clocks of a step or dispatch case."""
    n, R, pd, classes = case["rows"], case["replicas"], case["stages"] == "pd", _classes(case["classes"])
    t = _empty(n)
    rid = torch.arange(n, device="cuda") * R // n if case["layout"] == "grouped" else d.ints(0, R, n)
    t["replica_id"] = rid.to(torch.int32)
    share = torch.tensor({3: [1, 1, 1], 5: [1] * 5, 0: [3, 3, 2, 2], 4: [4, 3, 2, 1]}[case["classes"]], device="cuda", dtype=torch.float64)
    t["class_id"] = torch.bucketize(d.u(n), torch.cumsum(share / share.sum(), 0)[:-1]).to(torch.uint8)
    t["prompt_len"] = d.prompts(case["lengths"], n)
    t["output_len"] = d.lognormal(5.0, 0.8, 1, 2048, n)
    if case["weights"]:
        t["weight"] = d.ints(1, 17, n).to(torch.int32)
    if case["kind"] == "dispatch" or case["layout"] == "interleaved":
        now = torch.full((R,), NOW, dtype=torch.int64, device="cuda")      # one clock
    else:
        now = NOW + d.ints(0, SEC, R)
    now_r = now[rid]
    u = d.u(n)
    if case["future"] > 0:      # an arrival-ordered stream of a minute
        t["arrival_ns"] = torch.sort(NOW + _ns((d.u(n) - (1 - case["future"])) * 60 * SEC)).values
        age = torch.arange(n, device="cuda", dtype=torch.float64) / (n * (1 - case["future"]))
        come = t["arrival_ns"] <= now_r
        run = come & (age < (2 * case["inflight"] * d.u(R))[rid])      # the oldest ones of every instance are decoding
    else:                       # a backlog
        t["arrival_ns"] = now_r - _ns(d.exp(2.0, n) * SEC)
        come = torch.ones(n, dtype=torch.bool, device="cuda")
        run = u < case["inflight"]
    dec = rid >= R // 2
    if pd:
        per = n / R
        share_d = (d.u(R) * 256.0 / per).clamp(max=0.9)[rid]
        run = torch.where(dec, u < share_d, (u < 0.05 * case["inflight"] * (case["kind"] == "dispatch")))
        first = now_r - _ns(d.exp(0.05, n) * SEC)
        for k in ("first_token_ns", "last_token_ns"):
            t[k] = torch.where(dec, first, t[k])
        t["arrival_ns"] = torch.where(dec & come, torch.minimum(first - _ns((0.05 + 0.5 * d.u(n)) * SEC), t["arrival_ns"]), t["arrival_ns"])
    _in_flight(d, t, run, classes, now_r)
    if case["done"] > 0:
        _finished(d, t, come & ~run & (d.u(n) < case["done"]), classes, now_r)
    if case["ids"] == "permuted":
        t["req_id"] = d.permutation(n).to(torch.int32)
    reps = np.zeros((R, 3), np.int32)
    reps[:, 1] = 32768 if pd else 16384
    if pd:
        reps[:R // 2, 0], reps[R // 2:, 0], reps[R // 2:, 2] = W.PREFILL, W.DECODE, 256
    maturity = now - d.ints(0, 100 * MS, R)
    busy = d.u(R) < (0.125 if pd else 0.0)      # a batch is running
    maturity = torch.where(busy, now + d.ints(1 * MS, 400 * MS, R), maturity)
    return t, reps, now, maturity, classes


def _traces(case, d):
    """Columns of a batch of traces, rows sorted by arrival inside a trace, and the trace offsets."""
    T, m = case["traces"], case["rows"]
    lens = torch.full((T,), m, dtype=torch.int64, device="cuda")
    if case["ragged"]:
        lens = (d.u(T) * (m - m // 8) + m // 8).round().long().clamp(1, m)
    if case["bursty"]:      # two rates, re-drawn every 10 s
        periods = m // 50 + 8
        flip = (d.u(T, periods) < 0.5).long().cumsum(1) % 2
        rate = torch.where(flip == 1, 80.0, 5.0).to(torch.float64)
        edge = torch.cat([torch.zeros(T, 1, device="cuda", dtype=torch.float64), (rate * 10.0).cumsum(1)], 1)
        x = d.exp(1.0, T * m).view(T, m).cumsum(1)
        k = (torch.searchsorted(edge, x, right=True) - 1).clamp(max=periods - 1)
        arr = k * 10.0 + (x - edge.gather(1, k)) / rate.gather(1, k)
    else:
        arr = d.exp(1.0 / 20.0, T * m).view(T, m).cumsum(1)
    keep = torch.arange(m, device="cuda").unsqueeze(0) < lens.unsqueeze(1)
    arr = _ns(arr * SEC)[keep]
    n = arr.shape[0]
    t = _empty(n)
    t["arrival_ns"] = arr
    t["class_id"] = torch.bucketize(d.u(n), torch.tensor([0.4, 0.7, 0.9], device="cuda", dtype=torch.float64)).to(torch.uint8)
    t["prompt_len"] = d.prompts("lognormal", n)
    t["output_len"] = d.lognormal(5.0, 0.8, 1, 2048, n)
    off = np.zeros(T + 1, np.int32)
    off[1:] = np.cumsum(lens.cpu().numpy())
    return t, off


def _pd_table(case, d):
    """P instances 0 .. pairs - 1 and their partners in mid-run at one clock: old requests finished or decoding, some prefilled and in
    transfer, a backlog on the P side, the rest still to come (arrival order)."""
    n, pairs, classes = case["rows"], case["replicas"] // 2, W.CLASSES_PD
    t = _empty(n)
    p = d.ints(0, pairs, n)
    t["class_id"] = d.ints(0, len(classes), n).to(torch.uint8)
    t["prompt_len"] = d.lognormal(5.5, 1.0, 1, 4096, n)
    t["output_len"] = d.ints(1, 25, n).to(torch.int32)
    span = n / (40.0 * pairs)      # seconds, 40 requests/s per pair
    arr = torch.sort(NOW + _ns((d.u(n) - 0.5) * span * SEC)).values
    t["arrival_ns"] = arr
    age = (NOW - arr).to(torch.float64) / SEC
    done, on_d, on_p = age > 2.0, (age <= 2.0) & (age > 1.0), (age <= 1.0) & (age > 0.9)
    t["replica_id"] = torch.where(done | on_d, p + pairs, p).to(torch.int32)
    now_r = torch.full((n,), NOW, dtype=torch.int64, device="cuda")
    wait = on_d & (d.u(n) < 0.3)
    _finished(d, t, done, classes, now_r)
    _in_flight(d, t, on_d & ~wait, classes, now_r)
    t["first_token_ns"] = torch.where(on_p | wait, NOW - _ns(d.u(n) * 4 * MS), t["first_token_ns"])
    t["last_token_ns"] = torch.where(on_p | wait, t["first_token_ns"], t["last_token_ns"])
    t["state"] = torch.where(on_p, W.RUNNING, t["state"]).to(torch.uint8)
    if case["ids"] == "permuted":
        t["req_id"] = d.permutation(n).to(torch.int32)
    reps = np.zeros((2 * pairs, 3), np.int32)
    reps[:, 1] = 8192
    reps[:pairs, 0], reps[pairs:, 0], reps[pairs:, 2] = W.PREFILL, W.DECODE, 64
    now = torch.full((2 * pairs,), NOW, dtype=torch.int64, device="cuda")
    return t, reps, now, now - d.ints(0, 20 * MS, 2 * pairs), classes


def _elastic_table(case, d):
    """One global queue over a fleet in mid-run: the instances that are on hold what is decoding, new requests wait unbound."""
    n, R, classes = case["rows"], case["replicas"], W.CLASSES_4
    t = _empty(n)
    on = max(1, R // 8)
    t["class_id"] = torch.bucketize(d.u(n), torch.tensor([0.4, 0.7, 0.9], device="cuda", dtype=torch.float64)).to(torch.uint8)
    t["prompt_len"] = d.lognormal(6.0, 1.0, 16, 2000, n)
    t["output_len"] = d.ints(1, 25, n).to(torch.int32)
    arr = torch.sort(NOW + _ns((d.u(n) - 0.6) * n / (14.0 * on) * SEC)).values      # about what the instances that are on serve
    t["arrival_ns"] = arr
    age = (NOW - arr).to(torch.float64) / SEC
    done, run = age > 1.5, (age <= 1.5) & (age > 0.8)
    rid = torch.where(done | run, d.ints(0, on, n), -1)
    t["replica_id"] = rid.to(torch.int32)
    now_r = torch.full((n,), NOW, dtype=torch.int64, device="cuda")
    _finished(d, t, done, classes, now_r)
    _in_flight(d, t, run, classes, now_r)
    reps = np.zeros((R, 3), np.int32)
    reps[:, 1], reps[:, 2] = 8192, 64
    now = torch.full((R,), NOW, dtype=torch.int64, device="cuda")
    fleet = gen.new_fleet([4096] * R, range(on))
    fleet["since"][:on] = NOW
    fleet["due"][:on] = NOW
    return t, reps, now, now - d.ints(0, 20 * MS, R), classes, fleet


def prepare(case, seed):
    d, kind = _Draw(seed), case["kind"]
    s = dict(case=case)
    if kind == "sim":
        t, s["off"] = _traces(case, d)
        reps = np.zeros((case["traces"], 3), np.int32)
        reps[:, 1] = 16384
        s["table"] = hfx.DeviceTable(t)
        s["sched"] = hfx.Scheduler(W.DEFAULT_MODEL, W.CLASSES_4, reps, s["table"].n_rows, first_fit=case["first_fit"])
        s["out"] = hfx.SimOut(case["traces"])
        return s
    if kind == "monitor":
        n, w, P, m = case["rows"], case["window"], case["priorities"], case["requests"]
        t = _empty(n)
        t["class_id"] = d.ints(0, 4, n).to(torch.uint8)
        t["prompt_len"], t["output_len"] = d.prompts("lognormal", n), d.lognormal(5.0, 0.8, 1, 2048, n)
        t["arrival_ns"] = NOW - _ns(d.u(n) * 600 * SEC)
        _finished(d, t, d.u(n) < 0.9, W.CLASSES_4, torch.full((n,), NOW, dtype=torch.int64, device="cuda"))
        s["table"] = hfx.DeviceTable(t)
        s["sched"] = hfx.Scheduler(W.DEFAULT_MODEL, W.CLASSES_4, [[W.COLOCATED, 16384, 0]], n)
        s["att"] = torch.zeros((len(W.CLASSES_4) + 1, 6), dtype=torch.int64, device="cuda")
        s["window"] = dict(prio=d.ints(0, P, w).to(torch.int32), ttft_ns=_ns(torch.exp(-1.0 + d.normal(w)) * SEC), tpot_ns=_ns(torch.exp(-3.0 + 0.5 * d.normal(w)) * SEC),
                           queue_ns=_ns(d.exp(0.1, w) * SEC))
        p = torch.arange(P, device="cuda", dtype=torch.int64)
        s["bounds"] = dict(zip(SLO_BOUNDS, [x.contiguous() for x in (50 * MS * (p + 1), 2 * SEC * (p + 1), 100 * MS * (p + 1), 10 * MS * (p + 1), 60 * MS * (p + 1),
                                                                     20 * MS * (p + 1))]))
        s["last_queue"] = torch.zeros(P, dtype=torch.int64, device="cuda")
        s["pending"] = d.ints(0, 3, P).to(torch.int32)
        s["new_prio"] = d.ints(0, P, m).to(torch.int32)
        s["ttft"], s["tpot"] = (torch.zeros(m, dtype=torch.int64, device="cuda") for _ in range(2))
        return s
    opts = {}
    if kind == "pd":
        t, reps, s["now"], s["mat"], classes = _pd_table(case, d)
        s["pair"] = torch.from_numpy(W.pd_partner_table(case["replicas"] // 2)).cuda()
        s["moved"] = torch.zeros(4, dtype=torch.int32, device="cuda")
    elif kind == "elastic":
        t, reps, s["now"], s["mat"], classes, fleet = _elastic_table(case, d)
        s["fleet"] = hfx.Fleet(fleet)
        s["counts"] = torch.zeros((3, 4), dtype=torch.int64, device="cuda")
        s["used"] = torch.zeros(case["replicas"], dtype=torch.int64, device="cuda")
        s["decision"] = torch.zeros((3, 2), dtype=torch.int32, device="cuda")
        s["cost"] = torch.zeros(3, dtype=torch.int64, device="cuda")
        s["dout"] = hfx.DispatchOut(case["rows"], case["replicas"])
    else:
        t, reps, s["now"], s["mat"], classes = _table(case, d)
        opts = dict(budget_mode=hfx.BUDGET_CAP_ONLY if case["cap_only"] else hfx.BUDGET_SAFE, weight_max=16 if case["weights"] else 0,
                    first_fit=case["first_fit"])
    s["table"] = hfx.DeviceTable(t)
    s["sched"] = hfx.Scheduler(W.DEFAULT_MODEL, classes, reps, case["rows"], **opts)
    if kind == "dispatch":
        s["out"] = hfx.DispatchOut(case["rows"], case["replicas"])
    else:
        s["out"] = hfx.StepOut(case["rows"], case["replicas"], optional=case.get("outputs") == "all")
    if kind in ("pd", "elastic") or case.get("steps"):      # the snapshot that a pass starts from
        cols = MUTABLE + (("replica_id",) if kind != "step" else ())
        s["live"] = [t[k] for k in cols] + [s["now"], s["mat"]] + (list(s["fleet"].t.values()) if kind == "elastic" else [])
        s["snapshot"] = [x.clone() for x in s["live"]]
    return s


# ---- one pass ------------------------------------------------------------------------------------------------
def run(s):
    case, sched, table = s["case"], s["sched"], s["table"]
    kind = case["kind"]
    if kind == "sim":
        sched.sim_run(table, s["off"], case["iterations"], s["out"])
        return dict(s["out"].t, **{k: table.cols[k] for k in MUTABLE})
    if kind == "monitor":
        sched.attainment(table, s["att"])
        sched.slo_map(case["priorities"], s["window"], s["bounds"], s["last_queue"], s["pending"], s["new_prio"], s["ttft"], s["tpot"])
        return dict(attainment=s["att"], ttft=s["ttft"], tpot=s["tpot"], last_queue=s["last_queue"])
    if kind == "dispatch":
        sched.dispatch_step(table, NOW, s["mat"], s["out"])
        # (the library writes two numbers into n_queue and n_mature)
        return {k: v[:2] if k in ("n_queue", "n_mature") else v for k, v in s["out"].t.items()}
    now, mat, out = s["now"], s["mat"], s["out"]
    if kind == "step" and not case["steps"]:
        sched.step(table, now, mat, out)
        return {k: v for k, v in out.t.items() if v is not None}
    for x, y in zip(s["live"], s["snapshot"]):
        x.copy_(y)
    if kind == "step":
        for _ in range(case["steps"]):
            sched.step(table, now, mat, out, commit=True)
    elif kind == "pd":
        for _ in range(case["rounds"]):
            sched.step(table, now, mat, out, commit=True)
            sched.pd_migrate(table, now, mat, s["pair"], 2 * MS, 500, s["moved"])
    else:
        for k in range(case["rounds"]):
            now_g = NOW + (k + 1) * 50 * MS
            sched.set_horizon(now_g)
            for _ in range(6):
                sched.step(table, now, mat, out, commit=True)
            sched.scale_tick(table, now_g, s["fleet"].t["total_blocks"], s["counts"], s["used"], s["decision"], window_ns=2 * SEC)
            sched.scale_apply(now_g, s["decision"], s["used"], [300 * MS] * 3, s["fleet"], now, mat, s["cost"])
            sched.dispatch_step(table, now_g, s["fleet"].t["due"], s["dout"])
            sched.dispatch_bind(table, now_g, s["dout"], now)
    r = {k: v for k, v in out.t.items() if v is not None}
    r.update({k: table.cols[k] for k in MUTABLE}, now=now, maturity=mat)
    if kind == "pd":
        r.update(replica_id=table.cols["replica_id"], moved=s["moved"][:1])
    if kind == "elastic":
        r.update(replica_id=table.cols["replica_id"], counts=s["counts"], used=s["used"], decision=s["decision"], cost=s["cost"],
                 fleet=s["fleet"].t, assign=s["dout"].t["assign"], queue_order=s["dout"].t["queue_order"])
    return r


# ---- what a pass cannot do without ------------------------------------------------------------------------
# Bytes of the table's columns: replica 4, class 1, state 1, prompt 4, output length 4, gen 4, arrival 8, first / last token and finish 8
# each, id 4, weight 4.  "flops" are integer operations: about 30 per row for the latency model, slack and key, a comparison per level of
# the order, about 40 per simulated iteration.
def work(case):
    kind, n = case["kind"], case.get("rows", 0)
    if kind == "sim":
        rows = case["traces"] * case["rows"] * (0.5625 if case["ragged"] else 1)
        return dict(bytes=50 * rows, flops=case["traces"] * case["iterations"] * 40)
    if kind == "monitor":
        return dict(bytes=46 * n + 28 * case["window"] + 20 * case["requests"], flops=12 * n + 2 * case["window"] * math.log2(case["window"]) + 8 * case["requests"])
    R = case["replicas"]
    order = 30 + math.log2(max(2, n / R))
    step = 34 + 13                                      # columns in; slack, order and admit out
    if kind == "step":
        step += (4 if case["weights"] else 0) + (28 if case["outputs"] == "all" else 0)
        if not case["steps"]:
            return dict(bytes=step * n, flops=order * n)
        commit = 17 * case["inflight"]                  # output length in; state, gen and last token out, of the rows that decode
        return dict(bytes=n * (case["steps"] * (step + commit) + 58), flops=case["steps"] * order * n)
    dispatch = 34 + 16                                  # columns in; assignment, queue and slack out
    if kind == "dispatch":
        return dict(bytes=(dispatch + (4 if case["weights"] else 0)) * n, flops=(30 + math.log2(n)) * n)
    if kind == "pd":
        return dict(bytes=n * (case["rounds"] * (step + 14) + 66), flops=case["rounds"] * (order + 6) * n)
    return dict(bytes=n * (case["rounds"] * (6 * step + 30 + dispatch + 8) + 66), flops=case["rounds"] * (6 * order + 60) * n)


def tolerance(case):
    return "exact"
