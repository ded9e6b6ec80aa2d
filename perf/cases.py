"""The work this library is used for, as measurable cases.

Everything goes through the public entry points of ``paper_2602_11688_b200.binding``.  A case is a
dict of plain values; ``kind`` says which use it stands for:

  population  evaluate a population of weight vectors over an uploaded trace (the tuner's inner loop)
  scales      a load sweep: the population at every time scale, as one population
  windows     the rolling-window objective of the tuner on top of the population evaluation
  es          whole steps of the offline evolution strategy (host buffers in and out)
  online      the online tuner: weights change every hop inside one replay
  policies    the five baseline policies, one replay each
  extended    population evaluation with the optional model parts switched on
  live        the proxy's loop: requests are appended as they arrive, routed on a persistent state,
              and the decision is read back before the next batch
  upload      a new trace on the host is validated, prepared and copied to the GPU, and its first
              requests are routed

Traces come from the repository's own generator (``workloads.make_workload``) with its recipes;
``base`` names the recipe, the sizes are the case's.  Results are bit-exact by contract (routes, hits
and digests are integers; every time is fp64 in a fixed operation order), hence ``"exact"``.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2602_11688_b200 import binding as gb
from paper_2602_11688_b200 import workloads as W

FIRST_ROUTED = 1_000   # requests routed right after an upload

KINDS = ("population", "scales", "windows", "es", "online", "policies", "extended", "live", "upload")


def _case(name, kind, base, requests, population, *, replicas=None, slots=None, cache=None,
          detail=False, steps=0, batch=0, index=False, window=128, hop=32):
    """`cache` in blocks per replica (None: the recipe's share of a full-size trace, at least one
    longest prompt); `detail`: routes, hits and cache digests are wanted, not the p95s alone."""
    s = W.SPECS[base]
    if cache is None:
        cache = max(300, int(s.cache_blocks * requests / s.n_requests))
    return {"name": name, "kind": kind, "base": base, "requests": int(requests),
            "population": int(population), "replicas": int(replicas or s.n_replicas),
            "slots": int(slots or s.slots), "cache": int(cache), "detail": bool(detail),
            "steps": int(steps), "batch": int(batch), "index": bool(index),
            "window": int(window), "hop": int(hop)}


def listed():
    return [
        # the smallest configuration of the repository, whole: a quick look at a handful of weights
        _case("tiny population", "population", "tiny", 2_000, 8),
        # the multi-region configuration, whole, with everything a reader of the decisions asks for
        _case("regions population", "population", "regions", 50_000, 64, detail=True),
        # the headline workload (long prompts, high reuse) at a fifth of its requests, full population
        _case("longctx population", "population", "longctx", 100_000, 256, detail=True),
        # the largest fleet: 64 replicas x 64 slots, per-replica normalisers, more candidates than
        # the GPU has SMs for twice over; p95s alone, as a tuner asks for them
        _case("largest population", "population", "largest", 30_000, 400),
        # the saturation sweep: five load levels x 96 weight vectors as one population
        _case("sweep scales", "scales", "sweep", 30_000, 96),
        # objective of the tuner: p95 TTFT of 128-request windows every 32 requests
        _case("longctx windows", "windows", "longctx", 30_000, 100, window=128, hop=32),
        # four steps of the offline tuner with 16 offspring each
        _case("regions es", "es", "regions", 8_000, 16, steps=4),
        # the paper's tuner inside one replay, several start points side by side
        _case("tiny online tuner", "online", "tiny", 2_000, 8, steps=40),
        # the baselines a tuned weight vector is compared with
        _case("regions policies", "policies", "regions", 8_000, 1),
        # heterogeneous replicas, slow-down, KV budget, moving network, drifting index
        _case("longctx extended", "extended", "longctx", 12_000, 48, detail=True, index=True),
        # the proxy's loop, one request at a time: latency of a single decision
        _case("live one by one", "live", "regions", 192, 1, cache=400, batch=1),
        # a new trace comes in
        _case("longctx upload", "upload", "longctx", 40_000, 1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: use, recipe, and sizes spread over their whole range."""
    kind = rng.choice(KINDS)
    base = rng.choice(("regions", "longctx", "longctx", "sweep", "largest"))
    replicas = rng.choice((W.SPECS[base].n_replicas, _log_int(rng, 2, 64)))
    slots = rng.choice((W.SPECS[base].slots, _log_int(rng, 1, 64)))
    n = _log_int(rng, 1_500, 30_000)
    # caches from "evicts all the time" (a longest prompt) to "rarely full"
    cache = _log_int(rng, 300, 300 + n)
    kw = dict(replicas=replicas, slots=slots, cache=cache)
    if kind == "population":
        return _strip(_case("", kind, base, n, _log_int(rng, 1, 500), detail=rng.random() < 0.5, **kw))
    if kind == "scales":
        return _strip(_case("", kind, base, min(n, 20_000), _log_int(rng, 1, 90), **kw))
    if kind == "windows":
        window = rng.choice((128, _log_int(rng, 16, 1_000)))
        return _strip(_case("", kind, base, n, _log_int(rng, 1, 200), window=window,
                            hop=max(1, window // rng.choice((1, 4, 5))), **kw))
    if kind == "es":
        return _strip(_case("", kind, base, min(n, 12_000), _log_int(rng, 1, 64), steps=rng.randint(1, 5), **kw))
    if kind == "online":
        return _strip(_case("", kind, base, min(n, 6_000), _log_int(rng, 1, 64), steps=rng.randint(10, 150), **kw))
    if kind == "policies":
        return _strip(_case("", kind, base, min(n, 10_000), 1, **kw))
    if kind == "extended":
        # (the drifting index only where no prompt prefix is shared by a fifth of all requests)
        return _strip(_case("", kind, base, min(n, 15_000), _log_int(rng, 1, 100), detail=rng.random() < 0.5,
                            index=base != "regions" and rng.random() < 0.5, **kw))
    if kind == "live":
        batch = rng.choice((1, 1, _log_int(rng, 2, 64)))
        return _strip(_case("", kind, base, _log_int(rng, 100, 250) * min(batch, 16), 1, batch=batch, **kw))
    return _strip(_case("", kind, base, _log_int(rng, 2_000, 40_000), 1, **kw))


def _strip(case):
    return {k: v for k, v in case.items() if k != "name"}


def _workload(case, seed):
    """The recipe `base` with the case's sizes and another seed."""
    key = "%s at the sizes of a case" % case["base"]
    base = W.SPECS[case["base"]]
    R = case["replicas"]
    spec = dataclasses.replace(base, name=key, seed=int(seed), n_replicas=R, slots=case["slots"],
                               n_regions=min(base.n_regions, R), cache_blocks=case["cache"],
                               population=case["population"], n_requests=case["requests"],
                               n_sessions=max(1, case["requests"] // 10))
    W.SPECS[key] = spec
    try:
        return W.make_workload(key)
    finally:
        del W.SPECS[key]


def _ok(rc, where):
    if rc != gb.GORGO_OK:
        raise gb.GorgoError(rc, where)


def prepare(case, seed):
    """What a user's program holds before the call: the uploaded trace, the weights on the device,
    a workspace, output buffers.  (`upload`: the trace on the host; `live`: the trace on the host, a
    state and buffers on the device.)"""
    kind = case["kind"]
    w = _workload(case, seed)
    rng = np.random.default_rng(seed + 1)
    P, N, R, K = case["population"], w.n_requests, case["replicas"], w.n_params
    st = {"case": case, "w": w, "scale": float(w.spec.time_scales[0])}
    dev = torch.device("cuda", torch.cuda.current_device())
    if kind in ("upload", "live"):
        rc, st["h"] = gb.gorgo_sim_create(rtt_ms=w.rtt_ms, device=dev.index, **w.config_dict())
        _ok(rc, "gorgo_sim_create")
        rc, nbytes = gb.gorgo_trace_bytes(N, int(w.hash_off[-1]))
        _ok(rc, "gorgo_trace_bytes")
        st["buf"] = torch.empty(nbytes, dtype=torch.uint8, device=dev)
        st["stream"] = int(torch.cuda.current_stream(dev).cuda_stream)
        st["owner"] = _Handle(st["h"])
        st["params"] = np.ascontiguousarray(w.params[0])
        if kind == "live":
            st["batches"] = [_slice(w, a, min(N, a + case["batch"])) for a in range(0, N, case["batch"])]
            _ok(gb.gorgo_trace_begin(st["h"], N, int(w.hash_off[-1]), st["buf"]), "gorgo_trace_begin")
            _ok(gb.gorgo_trace_append(st["h"], *st["batches"][0][2], st["stream"]), "gorgo_trace_append")
        else:
            _upload_trace(st)
        rc, nbytes = gb.gorgo_state_bytes(st["h"])
        _ok(rc, "gorgo_state_bytes")
        st["state"] = torch.empty(nbytes, dtype=torch.uint8, device=dev)
        n = N if kind == "live" else min(N, FIRST_ROUTED)
        st["out"] = {"route": torch.empty(n, dtype=torch.uint8, device=dev),
                     "hit": torch.empty(n, dtype=torch.uint16, device=dev),
                     "ttft": torch.empty(n, dtype=torch.float64, device=dev),
                     "e2e": torch.empty(n, dtype=torch.float64, device=dev)}
        if kind == "live":
            st["h_route"] = torch.empty(N, dtype=torch.uint8).pin_memory()
        return st
    sim = gb.GorgoSim(w, device=dev.index)
    st["sim"], st["owner"] = sim, _Handle(sim.h)
    if kind == "extended":
        G = w.spec.n_regions
        _ok(gb.gorgo_sim_set_replica_speeds(sim.h, rng.uniform(0.03, 0.08, R), rng.uniform(15.0, 30.0, R)),
            "gorgo_sim_set_replica_speeds")
        _ok(gb.gorgo_sim_set_service_model(sim.h, 0.02, 32_000 * case["slots"]), "gorgo_sim_set_service_model")
        E = 40
        series = w.rtt_ms[None] * np.exp(np.cumsum(rng.normal(0.0, 0.1, size=(E, G, R)), axis=0))
        _ok(gb.gorgo_sim_set_rtt_series(sim.h, series, float(w.ts_ms[-1]) * st["scale"] / E, 0.3),
            "gorgo_sim_set_rtt_series")
        _ok(gb.gorgo_sim_set_proxy_index(sim.h, case["index"]), "gorgo_sim_set_proxy_index")
    if kind == "scales":
        scales = np.asarray(W.SPECS["sweep"].time_scales, dtype=np.float64)
        st["params"] = torch.from_numpy(np.tile(w.params, (len(scales), 1))).to(dev)
        st["scales"] = np.repeat(scales, P)
        P *= len(scales)
        st["route"] = torch.empty((P, N), dtype=torch.uint8, device=dev)
    elif kind == "windows":
        rc, n_win = gb.gorgo_window_count(N, case["window"], case["hop"])
        _ok(rc, "gorgo_window_count")
        st["params"] = torch.from_numpy(w.params).to(dev)
        st["win"] = torch.empty((P, n_win), dtype=torch.float64, device=dev)
        st["best"] = torch.empty(P, dtype=torch.float64, device=dev)
        st["which"] = torch.empty(P, dtype=torch.int32, device=dev)
    elif kind in ("es", "online"):
        x0 = np.ones(K)
        x0[0], x0[2] = 0.5, 0.1                              # start values and ranges of the paper
        st["es"] = dict(tuned=[0, 2], lo=[0.05, 0.05], hi=[2.0, 0.5], sigma0=0.5, sigma_up=1.5)
        if kind == "es":
            st["x0"], st["z"] = x0, rng.standard_normal((case["steps"], P, 2))
        else:
            st["x0"] = np.tile(x0, (P, 1)) * np.exp(rng.normal(0.0, 0.2, (P, 1)))
            st["z"] = rng.standard_normal((P, case["steps"], 2))
            st["route"] = torch.empty((P, N), dtype=torch.uint8, device=dev)
    elif kind == "policies":
        st["draws"] = rng.integers(0, 2 ** 32, size=N, dtype=np.uint32)
    sim.ensure_workspace(P)
    if kind in ("scales", "policies", "windows"):
        shape = (len(gb.POLICIES),) if kind == "policies" else (P,)
        st["p95_ttft"] = torch.empty(shape, dtype=torch.float64, device=dev)
        st["p95_e2e"] = torch.empty(shape, dtype=torch.float64, device=dev)
    if kind == "policies":
        st["route"] = torch.empty((len(gb.POLICIES), N), dtype=torch.uint8, device=dev)
        st["hit"] = torch.empty((len(gb.POLICIES), N), dtype=torch.uint16, device=dev)
    return st


class _Handle:
    """Destroys a simulator with the last reference to its state."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        gb.gorgo_sim_destroy(self.h)


def _slice(w, a, b):
    off = w.hash_off[a:b + 1]
    ids = w.hash_ids[int(off[0]):int(off[-1])]
    return a, b - a, (w.ts_ms[a:b], w.input_tokens[a:b], w.output_tokens[a:b], w.origin[a:b],
                      off - off[0], ids)


def run(state):
    return _RUN[state["case"]["kind"]](state)


def _population(st):
    d = st["case"]["detail"]
    out = st["sim"].eval_population(st["w"].params, st["scale"], want_route=d, want_hit=d, want_digest=d)
    if d:
        out["digest"] = out["digest"].view(torch.int64)
        out["hit"] = out["hit"].view(torch.int16)
    return out


def _scales(st):
    sim = st["sim"]
    _ok(gb.gorgo_eval_population_scales(sim.h, st["params"].shape[0], st["params"], st["scales"], sim.workspace,
                                        sim.stream, st["p95_ttft"], st["p95_e2e"], st["route"]), "scales")
    return st["p95_ttft"], st["p95_e2e"], st["route"]


def _windows(st):
    sim, c = st["sim"], st["case"]
    _ok(gb.gorgo_eval_population_windows(sim.h, c["population"], st["params"], st["scale"], sim.workspace,
                                         sim.stream, c["window"], c["hop"], st["win"], st["best"], st["which"],
                                         st["p95_ttft"], st["p95_e2e"]), "windows")
    return st["win"], st["best"], st["which"], st["p95_ttft"], st["p95_e2e"]


def _es(st):
    sim, c = st["sim"], st["case"]
    rc, x, f, sigma, hist = gb.gorgo_es_run(sim.h, x0=st["x0"], z=st["z"], n_steps=c["steps"], lam=c["population"],
                                            workspace=sim.workspace, stream=sim.stream,
                                            time_scale=st["scale"], **st["es"])
    _ok(rc, "gorgo_es_run")
    return x, f, sigma, hist


def _online(st):
    sim = st["sim"]
    rc, x, sigma, done, hist, pt, pe = gb.gorgo_tune_online(sim.h, x0=st["x0"], z=st["z"], workspace=sim.workspace,
                                                            stream=sim.stream, time_scale=st["scale"],
                                                            route=st["route"], **st["es"])
    _ok(rc, "gorgo_tune_online")
    return x, sigma, done, hist, pt, pe, st["route"]


def _policies(st):
    sim = st["sim"]
    for k, name in enumerate(gb.POLICIES):
        _ok(gb.gorgo_eval_policy(sim.h, name, st["draws"] if name == "random" else None, st["scale"],
                                 sim.workspace, sim.stream, st["p95_ttft"][k:], st["p95_e2e"][k:],
                                 st["route"][k], st["hit"][k]), name)
    return st["p95_ttft"], st["p95_e2e"], st["route"], st["hit"].view(torch.int16)


def _live(st):
    h, stream, out, state = st["h"], st["stream"], st["out"], st["state"]
    w = st["w"]
    _ok(gb.gorgo_trace_begin(h, w.n_requests, w.hash_ids.shape[0], st["buf"]), "gorgo_trace_begin")
    for a, n, arrays in st["batches"]:
        _ok(gb.gorgo_trace_append(h, *arrays, stream), "gorgo_trace_append")
        if a == 0:
            _ok(gb.gorgo_sim_reset(h, state, stream), "gorgo_sim_reset")
        _ok(gb.gorgo_route_batch(h, st["params"], st["scale"], a, n, state, stream, out["route"][a:],
                                 out["hit"][a:], out["ttft"][a:], out["e2e"][a:]), "gorgo_route_batch")
        st["h_route"][a:a + n].copy_(out["route"][a:a + n], non_blocking=True)
        torch.cuda.current_stream().synchronize()             # the proxy needs the decision now
    return st["h_route"], out["hit"].view(torch.int16), out["ttft"], out["e2e"]


def _upload_trace(st):
    w = st["w"]
    _ok(gb.gorgo_trace_upload(st["h"], w.ts_ms, w.input_tokens, w.output_tokens, w.origin, w.hash_off, w.hash_ids,
                              st["buf"], st["stream"]), "gorgo_trace_upload")


def _upload(st):
    h, out, state = st["h"], st["out"], st["state"]
    _upload_trace(st)
    _ok(gb.gorgo_sim_reset(h, state, st["stream"]), "gorgo_sim_reset")
    _ok(gb.gorgo_route_batch(h, st["params"], st["scale"], 0, out["route"].shape[0], state, st["stream"],
                             out["route"], out["hit"], out["ttft"], out["e2e"]), "gorgo_route_batch")
    return gb.gorgo_trace_info(h), out["route"], out["hit"].view(torch.int16), out["ttft"], out["e2e"]


_RUN = {"population": _population, "scales": _scales, "windows": _windows, "es": _es, "online": _online,
        "policies": _policies, "extended": _population, "live": _live, "upload": _upload}


def work(case):
    """Bytes: the trace (32 bytes of metadata per request, 8 per block id) and the weights read once,
    the results written once.  Flops: the score of every candidate, request and replica (three
    products, two sums)."""
    base = W.SPECS[case["base"]]
    N, R, P, kind = case["requests"], case["replicas"], case["population"], case["kind"]
    K = 3 + R if base.per_replica_normaliser else 3
    blocks = {"tiny": 12.5, "regions": 13.6}.get(case["base"], 59.0)   # mean blocks of a prompt
    replays = P
    if kind == "scales":
        replays = 5 * P
    elif kind == "es":
        replays = 1 + case["steps"] * P
    elif kind == "policies":
        replays = len(gb.POLICIES)
    elif kind == "upload":
        replays = 0
    nbytes = N * (32.0 + 8.0 * blocks) + replays * (8.0 * K + 16.0)
    if case["detail"] or kind == "policies":
        nbytes += replays * N * 3.0
    elif kind in ("online", "scales"):
        nbytes += replays * N
    elif kind == "live":
        nbytes += N * 19.0
    elif kind == "windows":
        nbytes += replays * 8.0 * max(0, (N - case["window"]) // case["hop"] + 1)
    elif kind == "upload":
        nbytes *= 2.0                                        # read on the host, written on the device
    return {"bytes": nbytes, "flops": 5.0 * replays * N * R}


def tolerance(case):
    return "exact"
