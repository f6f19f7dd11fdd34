"""What is measured: the calls a router's operator has this library make, from the smallest to the largest.

One case is one kind of work through the package's public entry points, on inputs that live on the GPU:

  hash      cr_hash_prefixes over one control interval's prefix spans (records padded to 16 bytes, or packed
            back to back as a tokenizer leaves them)
  plan      one turn of the control loop: the plans of every variant in use from the last interval's keys, then
            the interval's requests routed with them (the plan replicas only)
  live      one small batch of arriving requests dispatched on the running plan and the live loads
  route     one interval's requests routed for every (policy, seed) replica
  replay    one interval's routed requests through every LRU simulator, whose state carries over from pass to pass
            (capacities in prefixes, or in prefix tokens)
  interval  a whole control interval (hash, plan, route, replay) as the online driver takes it
  trace     the offline shadow replay of a trace of resident keys, optionally as a CUDA graph of the whole trace

Every output is a whole number and is compared exactly.
"""
import math

import numpy as np
import torch

import paper_2608_19677_gb300 as P
from paper_2608_19677_gb300.pipeline import TracePipeline, Pipeline

SIX = "CR,CR_NOLPT,CR_NOREPL,P2C,RR,HASH"
VARIANT = {"CR": "LPT", "CR_NOLPT": "RANDOM", "CR_NOREPL": "NOREPL", "CR_SLOTCAP": "SLOTCAP"}
WHALES = (3, 4, 5, 6, 7, 8, 9, 10)
SUFFIX = 64
VOCAB = 128256


def listed():
    return [
        # the 70B-shaped primary workload: one interval's prefix spans, the largest hash launch that fits beside others
        {"name": "hash_70b", "kind": "hash", "n": 166667, "median": 2048, "pmin": 16, "pmax": 16384, "align": 4},
        # a short interval of the 8B hot-key workload, spans packed back to back (any start offset)
        {"name": "hash_packed_8b", "kind": "hash", "n": 5000, "median": 0, "pmin": 1024, "pmax": 4096, "align": 1},
        # the hot-key study's control loop: small intervals, replicated keys, LPT next to three random placements
        {"name": "plan_8b", "kind": "plan", "n": 5000, "R": 16, "W": 64, "keys": 5000, "zipf": 1.1, "whales": True,
         "hot": False, "policies": "CR,CR_NOLPT", "seeds": 3, "B": 1024},
        # the large sweep's control loop: a million requests, ten plans
        {"name": "plan_large", "kind": "plan", "n": 1066667, "R": 1024, "W": 256, "keys": 1000000, "zipf": 0.8,
         "whales": False, "hot": False, "policies": "CR,CR_NOLPT,CR_NOREPL", "seeds": 8, "B": 1024},
        # online dispatch: a few hundred arrivals, each seeing every earlier one's load (latency and launches)
        {"name": "live_burst", "kind": "live", "n": 256, "R": 64, "W": 128, "keys": 100000, "zipf": 0.9,
         "whales": False, "hot": False, "policies": "CR", "seeds": 1, "B": 1, "planned": 133333},
        # the 70B-shaped comparison of four policies x five seeds, batched dispatch
        {"name": "route_70b", "kind": "route", "n": 166667, "R": 30, "W": 12, "keys": 20000, "zipf": 1.0,
         "whales": False, "hot": True, "policies": "CR,P2C,RR,HASH", "seeds": 5, "B": 1024},
        # exact sequential dispatch with the bounded-load policy beside CacheRoute and power-of-two choices
        {"name": "route_exact_70b", "kind": "route", "n": 83333, "R": 30, "W": 12, "keys": 20000, "zipf": 1.0,
         "whales": False, "hot": True, "policies": "CR,P2C,CHWBL", "seeds": 5, "B": 1},
        # bursty workload: 64 destinations, capacity 128, six policies x five seeds
        {"name": "replay_burst", "kind": "replay", "n": 133333, "R": 64, "W": 128, "keys": 100000, "zipf": 0.9,
         "whales": False, "hot": False, "policies": SIX, "seeds": 5, "caps": "128", "tokens": False, "median": 4096,
         "pmin": 16, "pmax": 32768},
        # the large sweep's interval: 1,024 destinations, 48 replicas, three capacities from one simulation
        {"name": "replay_large", "kind": "replay", "n": 1066667, "R": 1024, "W": 256, "keys": 1000000, "zipf": 0.8,
         "whales": False, "hot": False, "policies": SIX, "seeds": 8, "caps": "64,256,1024", "tokens": False,
         "median": 2048, "pmin": 16, "pmax": 32768},
        # the byte-aware replay of the 70B-shaped workload (24k-token budget per destination)
        {"name": "replay_tokens_70b", "kind": "replay", "n": 166667, "R": 30, "W": 12, "keys": 20000, "zipf": 1.0,
         "whales": False, "hot": True, "policies": "CR,P2C,RR,HASH", "seeds": 5, "caps": "24576", "tokens": True,
         "median": 2048, "pmin": 16, "pmax": 16384},
        # the smallest whole workload: one control interval, two policies
        {"name": "interval_tiny", "kind": "interval", "n": 20000, "R": 4, "W": 16, "keys": 200, "zipf": 1.1,
         "whales": False, "hot": False, "policies": "CR,P2C", "seeds": 1, "B": 1024, "caps": "16", "median": 0,
         "pmin": 512, "pmax": 512, "align": 4},
        # the large sweep as the offline gate runs it: several intervals in flight
        {"name": "trace_large", "kind": "trace", "n": 1066667, "intervals": 4, "R": 1024, "W": 256, "keys": 1000000,
         "zipf": 0.8, "whales": False, "hot": False, "policies": SIX, "seeds": 8, "B": 1024, "caps": "64,256,1024",
         "tokens": False, "median": 2048, "pmin": 16, "pmax": 32768, "group": 2, "graph": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["hash", "hash", "plan", "plan", "live", "route", "route", "replay", "replay", "interval",
                       "trace"])
    shape = rng.choice([(2048, 16, 16384), (4096, 16, 32768), (0, 1024, 4096), (0, 512, 512), (0, 1, 200)])
    lens = {"median": shape[0], "pmin": shape[1], "pmax": shape[2]}
    if kind == "hash":
        n = min(_log(rng, 8, 200000), int(4e8 / _mean_len(lens)))
        return {"kind": kind, "n": n, **lens, "align": rng.choice([4, 4, 2, 1])}
    R = _log(rng, 2, 1024)
    c = {"kind": kind, "R": R, "W": _log(rng, 2, 256), "keys": _log(rng, 100, 1000000),
         "zipf": rng.choice([0.8, 0.9, 1.0, 1.1]), "whales": rng.random() < 0.2, "hot": rng.random() < 0.3}
    if kind == "plan":
        return {**c, "n": _log(rng, 1000, 1066667), "seeds": rng.choice([1, 3, 8]),
                "policies": rng.choice(["CR", "CR,CR_NOLPT", "CR,CR_NOLPT,CR_NOREPL", "CR,CR_NOREPL,CR_SLOTCAP"]),
                "B": rng.choice([256, 1000, 1024])}
    if kind == "live":
        return {**c, "n": _log(rng, 1, 4096), "policies": rng.choice(["CR", "P2C", "CR_NOLPT", "CHWBL"]), "seeds": 1,
                "B": rng.choice([1, 1, 16, 64]), "planned": _log(rng, 1000, 200000)}
    pol = rng.choice(["CR,P2C", "CR,P2C,RR,HASH", "CR,CR_NOLPT,HASH,P2C", SIX])
    seeds = rng.choice([1, 3, 5, 8])
    pairs = 48 * 1066667 // (len(pol.split(",")) * seeds)
    if kind == "route":
        B = rng.choice([1, 7, 32, 333, 1024, 1024, 4096])
        if B <= 32:
            pol = rng.choice(["CR,P2C", "CR,P2C,CHWBL"])
        n = _log(rng, 1000, min(pairs, 1066667) if B > 32 else 150000)
        return {**c, "n": n, "policies": pol, "seeds": seeds, "B": B}
    caps = rng.choice(["12", "16", "64", "128", "8,32,100", "64,256,1024", "1024", "777"])
    if kind == "replay":
        tokens = rng.random() < 0.25
        if tokens:
            caps = rng.choice(["24576", "32768,131072", "524288"])
            c["R"] = _log(rng, 16, 1024)
        n = _log(rng, 1000, min(pairs, 200000 if tokens else 1066667))
        return {**c, "n": n, "policies": pol, "seeds": seeds, "caps": caps, "tokens": tokens, **lens}
    if kind == "interval":
        n = min(_log(rng, 1000, 100000), int(6e7 / (_mean_len(lens) + SUFFIX)))
        return {**c, "n": n, "policies": pol, "seeds": seeds, "B": 1024, "caps": caps, **lens,
                "align": rng.choice([4, 4, 1])}
    graph = rng.random() < 0.5
    n = _log(rng, 2000, 60000 if graph else 250000)
    T = rng.choice([3, 5, 8])
    return {**c, "n": n, "intervals": T, "policies": pol, "seeds": min(seeds, 5), "B": 1024, "caps": caps,
            "tokens": False, **lens, "group": rng.choice([1, 2, 4]), "graph": graph}


# ---- inputs --------------------------------------------------------------------------------------------------------

_ctx = None


def _context():
    """The program's library context, on the default stream."""
    global _ctx
    if _ctx is None:
        _ctx = P.Context(0)
    return _ctx


def _mean_len(case):
    if case["median"]:
        return case["median"] * math.exp(0.125)
    return (case["pmin"] + case["pmax"]) / 2.0


def _lens(case, n, g):
    """Prefix lengths: lognormal (sigma 0.5) around the median, or uniform, clamped."""
    if case["median"]:
        v = case["median"] * torch.exp(0.5 * torch.randn(n, generator=g, device="cuda"))
        return v.round().clamp(case["pmin"], case["pmax"]).to(torch.int32)
    return torch.randint(case["pmin"], case["pmax"] + 1, (n,), generator=g, device="cuda", dtype=torch.int32)


def _offsets(plen, align):
    """Record starts (prefix, suffix, padding to `align` tokens), packed in arrival order, and the arena's length."""
    rec = plen.to(torch.int64) + SUFFIX
    rec = (rec + align - 1) // align * align
    end = torch.cumsum(rec, 0)
    return end - rec, int(end[-1])


class _Workload:
    """Key popularity of a case: Zipf shares (optionally capped below the load target, optionally with injected hot
    keys), one random 64-bit routing key and one prefix length per business key."""

    def __init__(self, case, seed):
        self.case = case
        self.g = torch.Generator(device="cuda").manual_seed(seed)
        p = torch.arange(1, case["keys"] + 1, device="cuda", dtype=torch.float64) ** -case["zipf"]
        p /= p.sum()
        if case["hot"]:
            cap = max(0.8 / case["R"], 1.5 / case["keys"])
            for _ in range(40):
                over = p > cap
                excess = (p - cap).clamp(min=0).sum()
                p = torch.where(over, cap, p)
                free = torch.where(p < cap, p, 0.0)
                p = p + excess * free / free.sum().clamp(min=1e-30)
        if case["whales"]:
            w = torch.tensor(WHALES, device="cuda", dtype=torch.float64)
            p = torch.cat([0.75 * p / p.sum(), 0.25 * w / w.sum()])
        self.cdf = torch.cumsum(p / p.sum(), 0)
        self.K = int(p.shape[0])
        self.key = torch.randint(-(1 << 63), (1 << 63) - 1, (self.K,), generator=self.g, device="cuda")
        self.plen = _lens(case, self.K, self.g) if "median" in case else None

    def interval(self, n):
        u = torch.rand(n, generator=self.g, device="cuda", dtype=torch.float64)
        return torch.searchsorted(self.cdf, u, right=True).clamp(max=self.K - 1)

    def qcap(self, n):
        """Load target: 1.25 x the mean destination load, or (hot-key study) a fixed share of the interval."""
        return (max(n, 1), 208) if self.case["whales"] else (5 * max(n, 1), 4 * self.case["R"])


def _replicas(case):
    return [(p, s) for p in case["policies"].split(",") for s in range(case["seeds"])]


def _caps(case):
    return [int(c) for c in case["caps"].split(",")]


class _Routing:
    """The plans, rings and argument lists that routing every replica of a case takes."""

    def __init__(self, ctx, case, wl, keys):
        self.ctx, self.case = ctx, case
        reps = _replicas(case)
        self.policies = ["CR" if p == "CR_SLOTCAP" else p for p, _ in reps]
        self.seeds = [s for _, s in reps]
        kinds = []
        for p, s in reps:
            k = (VARIANT[p], s if p == "CR_NOLPT" else 0) if p in VARIANT else None
            if k is not None and k not in kinds:
                kinds.append(k)
        num, den = wl.qcap(int(keys.shape[0]))
        self.params = [P.plan_params(case["R"], case["W"], num, den, v, seed=s, epoch=1) for v, s in kinds]
        self.plans = [P.Plan(ctx) for _ in kinds]
        self.rep_plans = [self.plans[kinds.index((VARIANT[p], s if p == "CR_NOLPT" else 0))] if p in VARIANT else None
                          for p, s in reps]
        self.rings = [P.Ring(ctx, case["R"], 64, s) if p == "CHWBL" else None for p, s in reps]
        if self.plans:
            P.build_plans(ctx, keys, self.params, self.plans)

    def route(self, keys, g0, B, load, dest):
        return P.route_batch(self.ctx, self.rep_plans, self.policies, self.seeds, self.case["R"], keys, g0, B, load,
                             dest, rings=self.rings)


# ---- prepare -------------------------------------------------------------------------------------------------------

def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def _prepare_hash(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    plen = _lens(case, case["n"], g)
    off, total = _offsets(plen, case["align"])
    tok = torch.randint(0, VOCAB, (total,), generator=g, device="cuda", dtype=torch.int32)
    out = torch.empty(case["n"], dtype=torch.int64, device="cuda")
    return {"kind": "hash", "ctx": _context(), "tok": tok, "off": off, "plen": plen, "out": out, "salt": seed}


def _routed(case, seed, planned):
    """Plans from one interval's keys, another interval's keys, loads and destinations."""
    ctx, wl = _context(), _Workload(case, seed)
    prev = wl.key[wl.interval(planned)]
    kid = wl.interval(case["n"])
    n_rep = len(_replicas(case))
    s = {"kind": case["kind"], "ctx": ctx, "case": case, "wl": wl, "prev": prev, "kid": kid, "keys": wl.key[kid],
         "routing": _Routing(ctx, case, wl, prev), "g0": planned,
         "load": torch.zeros((n_rep, case["R"]), dtype=torch.int64, device="cuda"),
         "dest": torch.empty((n_rep, case["n"]), dtype=torch.int16, device="cuda")}
    return s


def _prepare_plan(case, seed):
    return _routed(case, seed, case["n"])


def _prepare_live(case, seed):
    s = _routed(case, seed, case["planned"])
    s["load"].copy_(torch.randint(0, 50, s["load"].shape, generator=s["wl"].g, device="cuda"))
    return s


def _prepare_route(case, seed):
    return _routed(case, seed, case["n"])


def _prepare_replay(case, seed):
    s = _routed(case, seed, case["n"])
    s["routing"].route(s["keys"], s["g0"], 1024, s["load"], s["dest"])
    s["plen"] = s["wl"].plen[s["kid"]]
    s["slen"] = torch.full_like(s["plen"], SUFFIX)
    n_rep, caps = len(_replicas(case)), _caps(case)
    s["replay"] = P.Replay(s["ctx"], n_rep, case["R"], caps, tokens=case["tokens"])
    s["ctr"] = torch.zeros((n_rep, len(caps), case["R"], 5), dtype=torch.int64, device="cuda")
    return s


def _prepare_interval(case, seed):
    ctx, wl = _context(), _Workload(case, seed)
    n = case["n"]
    kid = wl.interval(n)
    plen = wl.plen[kid]
    off, total = _offsets(plen, case["align"])
    # every token of a record from its key (prefix) or its request (suffix), so a key's requests share their prefix
    rec = torch.diff(off, append=torch.tensor([total], device="cuda"))
    req = torch.repeat_interleave(torch.arange(n, device="cuda"), rec)
    j = torch.arange(total, device="cuda") - off[req]
    stream = torch.where(j < plen[req], kid[req], wl.K + req)
    x = (stream * 1000003 + j * 7919 + seed % 1000003) % ((1 << 31) - 1)
    x = ((x * 48271 + 11) % ((1 << 31) - 1)) ^ (x >> 13)
    tok = (x % VOCAB).to(torch.int32)
    pipe = Pipeline(ctx, case["R"], case["W"], _caps(case), _replicas(case), wl.qcap, batch_B=case["B"], max_n=n)
    return {"kind": "interval", "pipe": pipe, "tok": tok, "off": off, "plen": plen,
            "slen": torch.full_like(plen, SUFFIX), "t": 0, "n": n}


def _prepare_trace(case, seed):
    wl = _Workload(case, seed)
    T = case["intervals"]
    # intervals of unequal size, as arrivals make them (the same for every seed, as the outputs' shapes are)
    sizes = [max(1, int(case["n"] * f)) for f in np.random.RandomState(case["n"] % 1000).uniform(0.97, 1.0, T)]
    kids = [wl.interval(m) for m in sizes]
    keys = [wl.key[k] for k in kids]
    plens = [wl.plen[k] for k in kids]
    slens = [torch.full_like(p, SUFFIX) for p in plens]
    g0s = [sum(sizes[:t]) for t in range(T)]
    stream = torch.cuda.Stream() if case["graph"] else torch.cuda.current_stream()
    stream.wait_stream(torch.cuda.current_stream())
    ctx = P.Context(0, stream) if case["graph"] else _context()
    pipe = TracePipeline(ctx, case["R"], case["W"], _caps(case), _replicas(case), wl.qcap, max_n=max(sizes),
                         batch_B=case["B"], depth=T, plan_streams=min(8, T), route_streams=min(4, T),
                         replay_group=case["group"])
    s = {"kind": "trace", "pipe": pipe, "in": (keys, plens, slens, g0s), "sizes": sizes, "ctx": ctx, "graph": None}
    pipe.reset()
    pipe.run(*s["in"])  # a running program's buffers
    pipe.quiesce()
    if case["graph"]:
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"], stream=stream):
            pipe.reset()
            pipe.run(*s["in"])
    return s


_PREPARE = {"hash": _prepare_hash, "plan": _prepare_plan, "live": _prepare_live, "route": _prepare_route,
            "replay": _prepare_replay, "interval": _prepare_interval, "trace": _prepare_trace}


# ---- run -----------------------------------------------------------------------------------------------------------

def run(state):
    return _RUN[state["kind"]](state)


def _run_hash(s):
    return P.hash_prefixes(s["ctx"], s["tok"], s["off"], s["plen"], s["salt"], out=s["out"])


def _run_plan(s):
    r = s["routing"]
    P.build_plans(s["ctx"], s["prev"], r.params, r.plans)
    s["load"].zero_()
    return [r.route(s["keys"], s["g0"], s["case"]["B"], s["load"], s["dest"]), s["load"]]


def _run_live(s):  # the live loads go on from pass to pass
    return [s["routing"].route(s["keys"], s["g0"], s["case"]["B"], s["load"], s["dest"]), s["load"]]


def _run_route(s):
    s["load"].zero_()
    return [s["routing"].route(s["keys"], s["g0"], s["case"]["B"], s["load"], s["dest"]), s["load"]]


def _run_replay(s):  # the simulators' state and the counters go on from pass to pass
    return P.shadow_replay(s["ctx"], s["replay"], s["keys"], s["plen"], s["slen"], s["dest"], s["ctr"])


def _run_interval(s):
    t = s["t"]
    s["t"] += 1
    pipe = s["pipe"]
    keys = pipe.interval(t, s["tok"], s["off"], s["plen"], s["slen"], t * s["n"])
    return {"keys": keys, "dest": pipe.last_dest, "ctr": pipe.ctr}


def _run_trace(s):
    pipe = s["pipe"]
    if s["graph"] is not None:
        s["graph"].replay()
    else:
        pipe.reset()
        pipe.run(*s["in"])
    return {"ctr": pipe.ctr, "dest": [pipe.dest_view(t, n) for t, n in enumerate(s["sizes"])]}


_RUN = {"hash": _run_hash, "plan": _run_plan, "live": _run_live, "route": _run_route, "replay": _run_replay,
        "interval": _run_interval, "trace": _run_trace}


# ---- work, tolerance -----------------------------------------------------------------------------------------------

def work(case):
    """Bytes of one pass: every input read once, every output written once."""
    n = case["n"]
    if case["kind"] == "hash":
        return {"bytes": n * (4 * _mean_len(case) + 8 + 4 + 8), "flops": 0}
    reps, R = len(_replicas(case)), case["R"]
    n_plans = len({(VARIANT[p], s if p == "CR_NOLPT" else 0) for p, s in _replicas(case) if p in VARIANT})
    adm = min(case["keys"], R * case["W"], n)
    table = 16 * adm + 2 * adm  # a key's slot and its member(s)
    route = 8 * n + 2 * n * reps + 16 * R * reps
    plan = 8 * n + n_plans * (table + 16 * min(case["keys"], n))
    replay = 0
    if "caps" in case:
        caps = _caps(case)
        held = 1024 if case.get("tokens") else max(caps)
        state = reps * R * min(held, n // R + 1) * (12 if case.get("tokens") else 8)
        replay = 16 * n + 2 * n * reps + 2 * state + 80 * reps * R * len(caps)
    kind = case["kind"]
    if kind == "plan":
        total = plan + route
    elif kind in ("live", "route"):
        total = route + n_plans * min(table, 18 * n)
    elif kind == "replay":
        total = replay
    elif kind == "interval":
        total = n * (4 * _mean_len(case) + 20) + plan + route + replay
    else:
        total = case["intervals"] * (plan + route + replay)
    return {"bytes": float(total), "flops": 0}


def tolerance(case):
    return "exact"


def exact(case, seed):
    """Every output is a whole number, held to the last bit by tolerance(): none has a value in floating point."""
    return None
