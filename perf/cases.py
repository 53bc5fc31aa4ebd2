"""Measured work of the routing library: what a user's program has it do, through its public entry points.

Kinds of case ("kind"):

  sim    simulate_replicas: a grid of closed-loop replicas over shared traces, with the Eq. (12) estimate
  hash   route_hash_blocks: block hashes of one ragged trace
  route  route_batch + route_release: a live router that routes batches and hears of the completions of earlier ones
  probe  route_probe: cached prefixes of a batch on every worker of a live router
  poa    poa_estimate: the windowed estimate on a caller's records
  knee   sweep_knee: percentiles and the saturation knee of concurrency sweeps on a caller's records

Every input is drawn from the seed alone.  Prompts have the workloads' shapes (lognormal lengths, shared-prefix
groups with Zipf popularity); a trace's tokens are produced on the device.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2606_17081_gb300 import routesim as rs
from paper_2606_17081_gb300 import streaming
from paper_2606_17081_gb300 import workloads as wk

DEV = "cuda"
MEAN_OVER_MEDIAN = math.exp(0.5 * 0.75 ** 2)   # of the lognormal prompt lengths (sigma 0.75)

# Fields of rs_replica_result that a simulation's user reads.  `probes`, `slow_path` and `rebuilds` count the
# library's own table operations, not anything of the simulated system, so they are no output here.
RESULT_FIELDS = [f for f, _ in rs.rs_replica_result._fields_ if f not in ("reserved0", "probes", "slow_path", "rebuilds")]


def _sim(name, grid, W, K, n_sim, n_traces, n_req, **more):
    c = {"name": name, "kind": "sim", "grid": grid, "W": W, "K": K, "n_sim": n_sim, "n_traces": n_traces, "n_req": n_req,
         "len_median": 1024, "len_max": 8192, "n_groups": 64, "variant": "lru", "records": True, "hashed": False, "C": 16}
    c.update(more)
    return c


def listed():
    return [
        # one short replica, the smallest call: launches, host steps and the serial event loop
        _sim("sim_tiny", "one", 3, 2048, 1, 1, 512, len_median=288, len_max=512, n_groups=16),
        # the 70B 1P/2D plan: a C sweep, selfish against load-balanced, caches that overflow; fewer replicas than SMs
        _sim("sim_p2d", "p2d", 3, 65536, 64, 7, 10000),
        # the parameter grid omega x C x tau with the coordinated policy beside every cell: more replicas than fit at once
        _sim("sim_grid", "grid", 6, 32768, 648, 3, 10000, records=False),
        # the 70B 1P/5D plan: adaptive controller and Eq. (2) sampling
        _sim("sim_p5d", "p5d", 6, 65536, 256, 18, 6000),
        # the 1P/2D plan under the KV Block Manager's frequency eviction
        _sim("sim_freq", "p2d", 3, 65536, 64, 7, 10000, variant="freq"),
        # 64 workers, prompts up to 32 768 tokens, traces given by their block hashes, a thousand in flight
        _sim("sim_wide", "wide", 64, 1 << 18, 16, 8, 5000, len_median=2048, len_max=32768, n_groups=1024, hashed=True, C=1024),
        # block hashing of a trace larger than L2
        {"name": "hash_trace", "kind": "hash", "n_req": 60000, "len_median": 1024, "len_max": 8192, "n_groups": 64},
        # a live router: one request at a time, as they come in ...
        {"name": "route_one", "kind": "route", "W": 6, "K": 8192, "batch": 1, "pool": 256, "tau": 0.0,
         "len_median": 1024, "len_max": 8192, "n_groups": 64},
        # ... and in batches
        {"name": "route_batch", "kind": "route", "W": 6, "K": 8192, "batch": 256, "pool": 8, "tau": 0.5,
         "len_median": 1024, "len_max": 8192, "n_groups": 64},
        # a batch probed against the caches of 64 workers
        {"name": "probe_wide", "kind": "probe", "W": 64, "K": 1 << 18, "routed": 2048, "n_req": 20000,
         "len_median": 2048, "len_max": 32768, "n_groups": 1024},
        # the PoA estimate of one replica's records, windows that bind the workers' capacity among them
        {"name": "poa_records", "kind": "poa", "W": 6, "n": 20000, "rate": 51.0},
        # the nine-level concurrency sweeps' percentiles and knees
        {"name": "knee_sweeps", "kind": "knee", "n_rep": 54, "levels": 9, "rows": 6000},
    ]


def _spread(rng, lo, hi):
    """A whole number in [lo, hi], uniform in its logarithm, seldom round."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["sim", "sim", "sim", "hash", "route", "probe", "poa", "knee"])
    if kind == "sim":
        if rng.random() < 0.25:   # many workers
            W = rng.randint(9, 64)
            c = _sim("", "wide", W, _spread(rng, 4096, 1 << 17), rng.randint(1, 16), 1, _spread(rng, 100, 3000), len_median=2048,
                     len_max=32768, n_groups=1024, hashed=rng.random() < 0.5, C=_spread(rng, 16, 1024))
        else:
            n_sim = _spread(rng, 1, 640)
            W = rng.randint(1, 8)
            waves = -(-n_sim // 304)
            c = _sim("", rng.choice(["one", "p2d", "p5d", "grid"]), W, _spread(rng, 1024, 65536), n_sim, 1,
                     _spread(rng, 100, 8000 // waves), len_median=_spread(rng, 128, 1024), n_groups=_spread(rng, 8, 256),
                     records=rng.random() < 0.5, C=_spread(rng, 1, 512))
            if rng.random() < 0.3 and c["grid"] in ("one", "p2d"):
                c["variant"] = rng.choice(["freq", "tiers"])
                if c["variant"] == "tiers":
                    c["W"] = min(W, 4)   # the tiers take W * (longest prompt's blocks) <= 2048
        c["n_traces"] = rng.randint(1, max(1, min(c["n_sim"], 12000 // c["n_req"], 8)))
        del c["name"]
        return c
    med = _spread(rng, 64, 2048)
    c = {"kind": kind, "len_median": med, "len_max": 8192, "n_groups": _spread(rng, 8, 512)}
    if kind == "hash":
        c["n_req"] = _spread(rng, 1, 60000 * 1024 // max(med, 1024))
    elif kind == "route":
        c.update(W=rng.randint(1, 64), K=_spread(rng, 1024, 65536), batch=_spread(rng, 1, 256), tau=rng.choice([0.0, 0.5, 1.0]))
        c["pool"] = max(2, min(64, 2048 // c["batch"]))
    elif kind == "probe":
        c.update(W=rng.randint(1, 64), K=_spread(rng, 1024, 1 << 17), routed=_spread(rng, 16, 1024), n_req=_spread(rng, 1, 16000))
    elif kind == "poa":
        return {"kind": kind, "W": rng.randint(2, 16) if rng.random() < 0.8 else rng.randint(17, 64), "n": _spread(rng, 64, 20000),
                "rate": float(rng.randint(10, 90))}
    else:
        return {"kind": kind, "n_rep": _spread(rng, 1, 128), "levels": rng.randint(1, 12), "rows": _spread(rng, 16, 20000)}
    return c


# ----------------------------------------------------------------- inputs

def _spec(c, n_req):
    tiny = c.get("grid") == "one" and c["len_max"] <= 512
    return wk.TraceSpec(n_req=n_req, len_kind="uniform" if tiny else "lognormal", len_median=float(c["len_median"]),
                        len_min=64 if tiny else 16, len_max=c["len_max"], n_groups=c["n_groups"],
                        prefix_min=min(256 if tiny else 512, c["len_max"]), prefix_max=min(256 if tiny else 2048, c["len_max"]),
                        zipf_s=None if tiny else 1.1, out_kind="uniform" if tiny else "lognormal", out_min=16 if tiny else 1,
                        out_max=256 if tiny else 4096, rate=50.0 if tiny else None, tokens="counter")


def _meta(c, n_req, seed, t=0):
    return wk.trace_meta(_spec(c, n_req), 1000 * int(seed) + t)


def _device_trace(meta):
    total = int(meta.offsets[-1])
    tokens = torch.zeros(total + (-total) % 4, dtype=torch.int32, device=DEV)
    meta.fill_device(meta.device(DEV), 0, total, tokens)
    return rs.TraceBuffers(tokens, torch.from_numpy(meta.offsets).to(DEV), torch.from_numpy(meta.release).to(DEV),
                           torch.from_numpy(meta.out_len).to(DEV), meta.n_req)


def _replicas(c):
    """The plan's replica list (the shapes of workloads.plan, cut to the case's sizes)."""
    reps = []
    for r in range(c["n_sim"]):
        t, n = r % c["n_traces"], c["n_req"]
        if c["grid"] == "p2d":
            sel = (r // 5) % 2 == 0
            rep = wk.Replica(t, [16, 32, 64, 128, 256][r % 5], wk.POLICY_DYNAMO if sel else wk.POLICY_LOADBAL, 0,
                             1.0 if sel else 0.0, 0.0, r // 10, n)
        elif c["grid"] == "p5d":
            cell = r % 15
            rep = wk.Replica(t, [32, 64, 128, 256, 512][cell % 5], wk.POLICY_DYNAMO, 1, 1.0, [0.0, 0.5, 1.0][cell // 5], r // 15, n)
        elif c["grid"] == "grid":
            cell = (r // 2) % 108
            C = [16, 32, 64, 128, 256, 512][(cell // 6) % 6]
            t = (r // 216) % c["n_traces"]
            if r % 2 == 0:
                rep = wk.Replica(t, C, wk.POLICY_DYNAMO, 0, [0.0, 0.25, 0.5, 1.0, 2.0, 4.0][cell % 6], [0.0, 0.5, 1.0][cell // 36], r // 216, n)
            else:
                rep = wk.Replica(t, C, wk.POLICY_LOADBAL, 0, 0.0, 0.0, r // 216, n)
        elif c["grid"] == "wide":
            sel = r < (c["n_sim"] + 1) // 2
            rep = wk.Replica(t, c["C"], wk.POLICY_DYNAMO if sel else wk.POLICY_LOADBAL, 0, 1.0 if sel else 0.0, 0.0, r, n)
        else:
            rep = wk.Replica(t, c["C"], wk.POLICY_DYNAMO, 0, 1.0, 0.0, r, n)
        if c["variant"] == "freq":
            rep.eviction, rep.freq_max, rep.decay_s = rs.RS_EVICT_FREQ, 64, 1.0
        reps.append(rep)
    return reps


class State:
    pass


def _prepare_sim(c, seed):
    s = State()
    more = {"tiered": 1, "tier_k2": c["K"], "tier_k3": 2 * c["K"]} if c["variant"] == "tiers" else {}
    s.ctx = rs.Context(W=c["W"], K=c["K"], stream=torch.cuda.current_stream().cuda_stream, **more)
    metas = [_meta(c, c["n_req"], seed, t) for t in range(c["n_traces"])]
    s.traces = [streaming.hash_streamed(s.ctx, m, device=DEV) if c["hashed"] else _device_trace(m) for m in metas]
    s.descs = [t.desc() for t in s.traces]
    s.params = [rs.replica_params(r) for r in _replicas(c)]
    s.rec = s.rec_t = None
    if c["records"]:
        s.rec, s.rec_t = rs.device_records(c["n_sim"] * c["n_req"], c["W"], device=DEV, with_cost=True, with_kv=c["variant"] == "tiers")
    return s


def _prepare_hash(c, seed):
    s = State()
    s.ctx = rs.Context(W=3, K=2048, stream=torch.cuda.current_stream().cuda_stream)
    s.trace = _device_trace(_meta(c, c["n_req"], seed))
    # room for any trace of these sizes (the sum's mean and seven times its spread); entries past the trace's stay 0
    room = min(c["n_req"] * c["len_max"], (c["n_req"] + 6 * math.sqrt(c["n_req"])) * _mean_len(c))
    s.out = torch.zeros(max(int(room), s.trace.tokens.numel()) // 16 + 1, dtype=torch.int64, device=DEV)
    return s


def _prepare_route(c, seed):
    """A router whose caches hold what earlier batches left, and the batches that come next."""
    s = State()
    n = c["batch"] * c["pool"]
    s.ctx = rs.Context(W=c["W"], K=c["K"], n_instances=1, stream=torch.cuda.current_stream().cuda_stream, tau=c["tau"], seed=int(seed))
    m = _meta(c, n, seed)
    s.trace = _device_trace(m)
    blocks = torch.from_numpy(((np.diff(m.offsets) + m.out_len + 15) // 16).astype(np.int32)).to(DEV)
    s.batches = [(s.trace.offsets[i:], s.trace.out_len[i:], blocks[i:i + c["batch"]].contiguous()) for i in range(0, n, c["batch"])]
    s.out = [(torch.zeros(c["batch"], dtype=torch.int32, device=DEV), torch.zeros(c["batch"], c["W"], device=DEV),
              torch.zeros(c["batch"], c["W"], dtype=torch.int32, device=DEV)) for _ in s.batches]
    s.n, s.k = c["batch"], 0
    for _ in range(c["pool"]):
        _run_route(s)
    return s


def _prepare_probe(c, seed):
    s = State()
    s.ctx = rs.Context(W=c["W"], K=c["K"], n_instances=1, stream=torch.cuda.current_stream().cuda_stream)
    s.trace = _device_trace(_meta(c, c["routed"] + c["n_req"], seed))
    worker = torch.zeros(c["routed"], dtype=torch.int32, device=DEV)
    rs.route_batch(s.ctx.h, 0, s.trace.tokens, s.trace.offsets, c["routed"], s.trace.out_len, worker)
    s.offsets = s.trace.offsets[c["routed"]:]
    s.n = c["n_req"]
    s.out = torch.zeros(s.n, c["W"], dtype=torch.int32, device=DEV)
    return s


def _records(c, seed):
    """Records of one replica as a run leaves them: Poisson arrivals, per-worker loads that drift, prefixes that a few workers
    hold per group, Eq. (9) latency with queueing on the busier workers, completion after the output tokens."""
    rng = np.random.default_rng([int(seed), 77])
    n, W = c["n"], c["W"]
    arrival = np.cumsum(rng.exponential(1.0 / c["rate"], n))
    arrival *= n / c["rate"] / arrival[-1]
    load = np.clip(24.0 + np.cumsum(rng.normal(0, 0.5, (n, W)), axis=0) + rng.normal(0, 6, W), 1, 63)
    n_frozen = np.minimum(np.rint(load) + 1, 63).astype(np.int16)
    L = np.clip(np.rint(np.exp(rng.normal(math.log(1024), 0.75, n))), 16, 8192).astype(np.int64)
    nbt = ((L + 15) // 16).astype(np.int32)
    group = np.minimum(rng.zipf(1.5, n) - 1, 63)
    held = rng.random((64, W)) < 0.4
    plen = rng.integers(32, 129, 64)
    prefix = np.where(held[group], np.minimum(plen[group], L // 16)[:, None], 0).astype(np.int16)
    worker = rng.integers(0, W, n).astype(np.int32)
    i = np.arange(n)
    nf, m = n_frozen[i, worker].astype(np.float64), prefix[i, worker].astype(np.float64)
    wait = np.where(nf >= 60, rng.exponential(2.0, n), 0.0)
    ttft = wait + (0.005 * nf + 0.020 + 0.010 / (64.0 - nf) ** 2) - 0.015 * m / nbt
    out = np.clip(np.rint(np.exp(rng.normal(math.log(256), 0.5, n))), 1, 4096)
    completion = np.minimum(arrival + ttft + 0.012 * out, n / c["rate"] + 50.0)
    completion[-1] = n / c["rate"] + 50.0   # the last request ends the run: every seed spans the same windows
    return {"worker": worker, "completion": completion, "ttft": ttft, "nbt": nbt,
            "n_frozen": n_frozen.reshape(-1), "prefix": prefix.reshape(-1)}


def _prepare_poa(c, seed):
    s = State()
    s.ctx = rs.Context(W=c["W"], K=2048, stream=torch.cuda.current_stream().cuda_stream)
    h = _records(c, seed)
    s.t = {k: torch.from_numpy(v).to(DEV) for k, v in h.items()}
    s.rec = rs.rs_records(*[s.t[k].data_ptr() if k in s.t else None for k, _ in rs.rs_records._fields_])
    s.n, s.cap = c["n"], int(h["completion"].max() / 5.0) + 2
    return s


def _sweep_inputs(c, seed):
    rng = np.random.default_rng([int(seed), 78])
    nr = c["n_rep"]
    load = np.array([2.0 ** (r % c["levels"]) for r in range(nr)])
    start = np.array(sorted({*range(0, nr, c["levels"]), nr}), np.int32)
    rows = c["rows"]
    mean = 0.05 + 0.004 * load + np.maximum(0.0, load - 48.0) ** 1.5 * 0.01   # flat, then queueing past saturation
    ttft = (mean[:, None] * np.exp(rng.normal(0, 0.4, (nr, rows)))).reshape(-1)
    return load, start, np.arange(nr + 1, dtype=np.int64) * rows, ttft


def _prepare_knee(c, seed):
    s = State()
    s.ctx = rs.Context(W=3, K=2048, stream=torch.cuda.current_stream().cuda_stream)
    s.load, s.start, s.rows, ttft = _sweep_inputs(c, seed)
    s.ttft = torch.from_numpy(ttft).to(DEV)
    s.worker = torch.zeros(ttft.size, dtype=torch.int32, device=DEV)
    s.rec = rs.rs_records(worker=s.worker.data_ptr(), ttft=s.ttft.data_ptr())
    return s


def prepare(case, seed):
    s = {"sim": _prepare_sim, "hash": _prepare_hash, "route": _prepare_route, "probe": _prepare_probe, "poa": _prepare_poa,
         "knee": _prepare_knee}[case["kind"]](case, seed)
    s.kind = case["kind"]
    return s


# ----------------------------------------------------------------- one pass

def _run_route(s):
    offs, out_len, _ = s.batches[s.k]
    worker, cost, prefix = s.out[s.k]
    rs.route_batch(s.ctx.h, 0, s.trace.tokens, offs, s.n, out_len, worker, cost, prefix)
    before = (s.k - 1) % len(s.batches)   # the batch before this one has completed (at first: zeros, no load is left below 0)
    rs.route_release(s.ctx.h, 0, s.out[before][0], s.batches[before][2], s.n)
    s.k = (s.k + 1) % len(s.batches)
    return {"worker": worker, "cost": cost, "prefix": prefix}


def run(s):
    if s.kind == "sim":
        res = rs.simulate_replicas(s.ctx.h, s.descs, rs.RS_MEM_DEVICE, s.params, s.rec)
        r = np.ctypeslib.as_array(res)
        return {"results": {f: r[f] for f in RESULT_FIELDS}, "records": s.rec_t}
    if s.kind == "hash":
        rs.route_hash_blocks(s.ctx.h, s.trace.tokens, s.trace.offsets, s.trace.n_req, s.out)
        return s.out
    if s.kind == "route":
        return _run_route(s)
    if s.kind == "probe":
        rs.route_probe(s.ctx.h, 0, s.trace.tokens, s.offsets, s.n, s.out)
        return s.out
    if s.kind == "poa":
        numer, opt, count, total, nw = rs.poa_estimate(s.ctx.h, s.rec, s.n, s.cap)
        return {"numer": numer, "opt": opt, "count": count, "total": total, "windows": nw}
    return rs.sweep_knee(s.ctx.h, s.rec, s.rows, s.load, s.start)


# ----------------------------------------------------------------- what a pass cannot do without

def _mean_len(c):
    return 288.0 if c.get("grid") == "one" and c["len_max"] <= 512 else min(c["len_median"] * MEAN_OVER_MEDIAN, c["len_max"])


def work(case):
    """Bytes of the inputs read once and the outputs written once; the integer work of hashing and the float64 work of the
    estimate are a few operations per byte and left at 0."""
    c, k = case, case["kind"]
    if k == "sim":
        req = c["n_traces"] * c["n_req"]
        tokens = req * _mean_len(c)
        inputs = (tokens / 2 if c["hashed"] else 4 * tokens) + req * 20
        per_row = 48 + 8 * c["W"] + (8 if c["variant"] == "tiers" else 0) if c["records"] else 0
        return {"bytes": inputs + c["n_sim"] * (c["n_req"] * per_row + ctypes.sizeof(rs.rs_replica_result)), "flops": 0}
    if k == "hash":
        return {"bytes": c["n_req"] * (4.5 * _mean_len(c) + 8), "flops": 0}
    if k == "route":
        return {"bytes": c["batch"] * (4 * _mean_len(c) + 24 + 8 * c["W"]), "flops": 0}
    if k == "probe":
        return {"bytes": c["n_req"] * (4 * _mean_len(c) + 8 + 4 * c["W"]), "flops": 0}
    if k == "poa":
        return {"bytes": c["n"] * (24 + 4 * c["W"]) + c["n"] / c["rate"] / 5 * 24, "flops": 0}
    return {"bytes": c["n_rep"] * (12 * c["rows"] + 40), "flops": 0}


def tolerance(case):
    """Decisions, prefixes, hashes, loads and event times are determined by the method operation by operation.  Sums over
    records may be taken in another order: 64-bit sums.  OPT's optimum is unique, its summands are not (equal-cost
    assignments), and the solvers ignore gains below 1e-12."""
    if case["kind"] in ("hash", "route", "probe"):
        return "exact"
    if case["kind"] == "knee":
        return {"rel": 1e-14, "max": 1e-13}
    return {"rel": 1e-12, "max": 1e-11}


# ----------------------------------------------------------------- the same in plain numpy

def _opt(cost, cap):
    """Least cost of assigning every row of cost [m, W] to a worker, at most cap rows each: rows start at their cheapest
    worker; those past a capacity are taken out and put back along shortest augmenting paths."""
    m, W = cost.shape
    at = cost.argmin(1)
    count = np.bincount(at, minlength=W)
    if (count <= cap).all():
        return float(cost[np.arange(m), at].sum())
    for j in range(W):
        rows = np.nonzero(at == j)[0]
        at[rows[cap:]] = -1
    count = np.minimum(count, cap)
    for r0 in np.nonzero(at < 0)[0]:
        edge, row = np.full((W, W), np.inf), np.zeros((W, W), np.int64)
        for j in range(W):
            rows = np.nonzero(at == j)[0]
            if rows.size:
                d = cost[rows] - cost[rows, j:j + 1]
                best = d.argmin(0)
                edge[j], row[j] = d[best, np.arange(W)], rows[best]
                edge[j, j] = np.inf
        dist, pred = cost[r0].copy(), np.full(W, -1)
        for _ in range(W):
            via = dist[:, None] + edge
            j = via.argmin(0)
            v = via[j, np.arange(W)]
            better = v < dist - 1e-13
            if not better.any():
                break
            dist, pred = np.where(better, v, dist), np.where(better, j, pred)
        k = int(np.where(count < cap, dist, np.inf).argmin())
        count[k] += 1
        while pred[k] >= 0:
            j = int(pred[k])
            at[row[j, k]] = k
            k = j
        at[r0] = k
    return float(cost[np.arange(m), at].sum())


def _exact_poa(worker, completion, ttft, nbt, n_frozen, prefix, W):
    nf, m = n_frozen.reshape(-1, W).astype(np.float64), prefix.reshape(-1, W).astype(np.float64)
    cost = 0.005 * nf + 0.020 + 0.010 / (64.0 - nf) ** 2 - 0.015 * m / np.maximum(nbt, 1)[:, None]
    win = np.floor(completion / 5.0).astype(np.int64)
    nw = int(win.max()) + 1
    numer, opt, count = np.zeros(nw), np.zeros(nw), np.zeros(nw, np.int64)
    for w in range(nw):
        rows = np.nonzero(win == w)[0]
        if rows.size:
            numer[w], count[w] = math.fsum(ttft[rows]), rows.size
            opt[w] = _opt(cost[rows], max(64, -(-rows.size // W)))
    return numer, opt, count, math.fsum(numer) / math.fsum(opt)


def _exact_sim(c, seed):
    """One replica of the closed loop at tau = 0 under LRU: caches as ordered dicts keyed by prompt content."""
    meta = _meta(c, c["n_req"], seed)
    tr, rep, W, K = meta.trace(c["n_req"]), _replicas(c)[0], c["W"], c["K"]
    cache = [dict() for _ in range(W)]
    active, serving, queue = [0] * W, [0] * W, [[] for _ in range(W)]
    n = c["n_req"]
    rec = {k: np.zeros(n) for k in ("arrival", "start", "first_token", "completion", "ttft")}
    worker, nbt_a = np.zeros(n, np.int64), np.zeros(n, np.int64)
    nfz, pre = np.zeros((n, W)), np.zeros((n, W))
    events, wco, blk = [], np.zeros(n), np.zeros(n, np.int64)
    inflight, prev = 0, 0.0

    def start(i, t):
        j = worker[i]
        serving[j] += 1
        k = serving[j]
        rec["start"][i] = t
        rec["first_token"][i] = t + (0.005 * k + 0.020 + 0.010 / (64.0 - k) ** 2 - wco[i])
        rec["ttft"][i] = rec["first_token"][i] - rec["arrival"][i]
        rec["completion"][i] = rec["first_token"][i] + tr.out_len[i] * 0.012
        events.append((rec["completion"][i], i))
        events.sort(reverse=True)

    def finish():
        nonlocal inflight
        t, i = events.pop()
        j = worker[i]
        serving[j] -= 1
        active[j] -= blk[i]
        inflight -= 1
        if queue[j]:
            start(queue[j].pop(0), t)
        return t

    for i in range(n):
        tok = tr.tokens[tr.offsets[i]:tr.offsets[i + 1]]
        L, nb = tok.size, tok.size // 16
        keys, h = [], b""
        for k in range(nb):
            h = hash((h, tok[16 * k:16 * k + 16].tobytes()))
            keys.append(h)
        t = prev
        while inflight >= rep.C:
            t = max(t, finish())
        t = max(t, tr.release[i])
        while events and events[-1][0] <= t:
            finish()
        prev = rec["arrival"][i] = t
        nbt_a[i] = (L + 15) // 16
        cost = []
        for j in range(W):
            m = 0
            while m < nb and keys[m] in cache[j]:
                m += 1
            pre[i, j], nfz[i, j] = m, min(serving[j] + 1, 63)
            cost.append(rep.omega * (nbt_a[i] - m) + active[j])
        j = int(np.argmin(cost))
        worker[i] = j
        for key in keys:
            if key in cache[j]:
                del cache[j][key]
            elif len(cache[j]) >= K:
                del cache[j][next(iter(cache[j]))]
            cache[j][key] = None
        wco[i] = 0.015 * (pre[i, j] / max(nbt_a[i], 1))
        blk[i] = (L + tr.out_len[i] + 15) // 16
        active[j] += blk[i]
        inflight += 1
        if serving[j] < 63:
            start(i, t)
        else:
            queue[j].append(i)
    while events:
        finish()
    total = _exact_poa(worker, rec["completion"], rec["ttft"], nbt_a, nfz.reshape(-1), pre.reshape(-1), W)[3]
    res = {"sum_ttft": math.fsum(rec["ttft"]), "sum_e2e": math.fsum(rec["completion"] - rec["arrival"]),
           "makespan": rec["completion"].max(), "poa_total": total}
    return {"results": {k: np.array([v]) for k, v in res.items()}, "records": rec}


def exact(case, seed):
    """float64 values of the estimates and of a small simulation; decisions, hashes and prefixes are whole numbers."""
    c, k = case, case["kind"]
    if k == "sim" and c["grid"] == "one" and c["variant"] == "lru" and c["n_sim"] == 1 and c["n_req"] <= 1000:
        return _exact_sim(c, seed)
    if k == "poa" and c["W"] <= 16:
        numer, opt, count, total = _exact_poa(*[_records(c, seed)[f] for f in ("worker", "completion", "ttft", "nbt", "n_frozen", "prefix")],
                                              c["W"])
        return {"numer": numer, "opt": opt, "count": count, "total": total, "windows": numer.size}
    if k == "knee":
        load, start, rows, ttft = _sweep_inputs(c, seed)
        v = np.sort(ttft.reshape(c["n_rep"], -1), axis=1)
        stat = v[:, (99 * c["rows"] + 99) // 100 - 1]
        d1, d2 = np.full(c["n_rep"], np.nan), np.full(c["n_rep"], np.nan)
        for a, b in zip(start[:-1], start[1:]):
            for r in range(a, b - 1):
                d1[r] = (stat[r + 1] - stat[r]) / (load[r + 1] - load[r])
            for r in range(a + 1, b - 1):
                d2[r] = 2.0 * (d1[r] - d1[r - 1]) / (load[r + 1] - load[r - 1])
        return {"stat": stat, "d1": d1, "d2": d2}
    return None
