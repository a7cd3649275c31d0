"""The Estimator's work as its users have it done, case by case, through the public entry points.

A case names an entry point, a pipeline, a trace and a set of candidate configurations:

  call       "estimate"   P99 and misses of every candidate; entry "host" (numpy in and out, as a Planner process
                          calls it) or "device" (torch tensors that stay on the GPU)
             "feasible"   only whether P99 meets the objective, host or device
             "latencies"  the latency of every query for one configuration
             "plan"       a whole Planner run (Algorithms 1 and 2), a few to some twenty calls that depend on each other
             "envelope"   the traffic envelope of the trace, Planner to Tuner
  pipeline   "chain" of `stages` models, "tree6" / "tree8" (conditional branches), "fanout6" (parallel branches),
             "diamond" (two branches that join)
  space      where the candidates come from: "random" draws over the whole grid of hardware, batch and replicas;
             "step", the questions of one Planner iteration (all candidates are one model away from one plan);
             "product", an exhaustive sweep over per-stage choices

Traces are Gamma renewal processes given by rate and CV or a ramp of the rate, tables are affine in the batch: the
shapes of the repository's five workloads, seeded afresh for every state.
"""
import math

import numpy as np
import torch

import paper_1812_01776_b200 as il
from paper_1812_01776_b200.planner import Planner, envelope_windows
from workloads import (affine_tables, bernoulli_bits, gamma_arrivals, product_candidates, ramp_arrivals,
                       uniform_candidates)

# pipeline: parent, guard bit, guard value per stage, second incoming edge, probability of each branch bit
_PIPES = {
    "tree6": ([-1, 0, 1, 0, 3, 4], [-1, 0, -1, 0, -1, -1], [0, 0, 0, 1, 0, 0], None, [0.7]),
    "tree8": ([-1, 0, 0, 1, 1, 2, 2, 3], [-1, 0, 0, 1, 1, 2, 2, -1], [0, 0, 1, 0, 1, 0, 1, 0], None, [0.5, 0.3, 0.7]),
    "fanout6": ([-1, 0, 0, 1, 2, 2], [-1, -1, -1, -1, 0, -1], [0, 0, 0, 0, 1, 0], None, [0.5]),
    "diamond": ([-1, 0, 0, 1], [-1] * 4, [0] * 4, [-1, -1, -1, 2], []),
}


def _case(call, entry, pipeline, stages, hw, max_batch, replicas, queries, qps, cv, candidates, space, slo_us, **more):
    return dict(call=call, entry=entry, pipeline=pipeline, stages=stages, hw=hw, max_batch=max_batch, replicas=replicas,
                queries=queries, qps=qps, cv=cv, candidates=candidates, space=space, slo_us=slo_us, **more)


def listed():
    return [
        # the smallest question: a two-stage pipeline, a short trace, a handful of candidates (workload 1 in full)
        _case("estimate", "host", "chain", 2, 2, 16, 4, 2_000, 100.0, 1.0, 64, "random", 150_000, name="small_batch"),
        # one iteration of the Planner on an image pipeline: about a thousand neighbours of one plan
        _case("estimate", "host", "chain", 4, 3, 32, 8, 50_000, 200.0, 4.0, 903, "step", 200_000, name="planner_step"),
        # what a Planner user waits for: all of its calls, on a trace of half the length
        _case("plan", "host", "chain", 4, 3, 32, 8, 25_000, 200.0, 4.0, 1, "step", 200_000, name="planner_run"),
        # a batch of unrelated candidates on the image pipeline (workload 2 in full)
        _case("estimate", "device", "chain", 4, 3, 32, 8, 50_000, 200.0, 4.0, 4_096, "random", 200_000, name="chain4"),
        # a large batch on a pipeline with a conditional branch, odd sizes (workload 3's shape)
        _case("estimate", "device", "tree6", 6, 3, 64, 8, 199_999, 300.0, 1.0, 7_001, "random", 250_000, name="tree6"),
        # the largest: 1.4 hours of a ramping trace through ten stages (workload 4's shape)
        _case("estimate", "device", "chain", 10, 4, 64, 16, 1_000_000, 150.0, 0.0, 4_096, "random", 300_000,
              name="chain10_long"),
        # an exhaustive sweep over per-stage choices (workload 5 in full: 2^20 candidates)
        _case("estimate", "device", "tree8", 8, 4, 64, 32, 100_000, 500.0, 2.0, 1 << 20, "product", 200_000,
              choices="8,8,8,8,4,4,4,4", name="sweep_tree8"),
        # the Planner's question alone, a large batch on a tree
        _case("feasible", "device", "tree6", 6, 3, 64, 8, 100_000, 300.0, 1.0, 8_192, "random", 250_000,
              name="feasible_tree6"),
        # parallel branches
        _case("estimate", "device", "fanout6", 6, 2, 16, 8, 100_000, 300.0, 2.0, 2_048, "random", 200_000, name="fan_out"),
        # branches that join
        _case("estimate", "host", "diamond", 4, 2, 16, 8, 50_000, 300.0, 2.0, 511, "random", 200_000, name="join"),
        # the latency of every query under one configuration, as for a plot of it
        _case("latencies", "host", "chain", 4, 3, 32, 8, 50_000, 200.0, 4.0, 1, "random", 200_000, name="one_config"),
        # traffic envelope of a long trace, as the Planner hands it to the Tuner
        _case("envelope", "host", "chain", 4, 3, 32, 8, 1_000_000, 200.0, 4.0, 1, "random", 200_000, name="envelope"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["estimate"] * 6 + ["feasible"] * 2 + ["sweep", "fan", "join", "latencies", "plan", "envelope"])
    queries = _log(rng, 1_000, 400_000)
    entry = rng.choice(["host", "device"])
    hw, replicas = rng.randint(2, 4), rng.choice([4, 8, 16, 32])
    max_batch, cv = rng.choice([8, 16, 32, 33, 64]), rng.choice([1.0, 2.0, 4.0])
    qps, slo = round(rng.uniform(100.0, 500.0), 1), rng.choice([150_000, 200_000, 250_000, 300_000])
    common = dict(hw=hw, max_batch=max_batch, replicas=replicas, qps=qps, cv=cv, slo_us=slo)
    if kind == "sweep":
        k = [rng.randint(2, 8) for _ in range(8)]
        return _case("estimate", entry, "tree8", 8, queries=min(queries, 150_000), candidates=math.prod(k), space="product",
                     choices=",".join(map(str, k)), **common)
    if kind == "fan":
        queries = min(queries, 100_000)
        return _case("estimate", entry, "fanout6", 6, queries=queries, candidates=_log(rng, 32, 2_048), space="random", **common)
    if kind == "join":
        queries = min(queries, 50_000)
        return _case("estimate", entry, "diamond", 4, queries=queries, candidates=_log(rng, 16, 511), space="random", **common)
    if kind in ("latencies", "envelope"):
        return _case(kind, "host", "chain", rng.randint(1, 10), queries=queries, candidates=1, space="random", **common)
    if kind == "plan":
        common.update(replicas=8, qps=200.0, slo_us=200_000, hw=3, max_batch=32)
        return _case("plan", "host", "chain", rng.randint(3, 4), queries=_log(rng, 2_000, 25_000), candidates=1, space="step",
                     **common)
    pipeline = rng.choice(["chain", "chain", "tree6", "tree8"])
    stages = rng.randint(1, 12) if pipeline == "chain" else len(_PIPES[pipeline][0])
    # at most a quarter of the largest listed case's query-events
    most = max(16, min(16_384, int(1e10 / (queries * stages))))
    space = rng.choice(["random", "random", "step"])
    candidates = _log(rng, 16, min(most, 2_048) if space == "step" else most)
    return _case(kind, entry, pipeline, stages, queries=queries, candidates=candidates, space=space, **common)


def _pipe(case):
    S = case["stages"]
    if case["pipeline"] == "chain":
        return list(range(-1, S - 1)), [-1] * S, [0] * S, None, []
    return _PIPES[case["pipeline"]]


def _visits(case):
    """Expected share of the queries that visits each stage, and copies of a query that leave."""
    parent, bit, val, parent2, probs = _pipe(case)
    share = [1.0] * len(parent)
    for s in range(1, len(parent)):
        p = 1.0 if bit[s] < 0 else (probs[bit[s]] if val[s] else 1.0 - probs[bit[s]])
        share[s] = share[parent[s]] * p
    return share


def _tables(case, rng):
    S, H, B = case["stages"], case["hw"], case["max_batch"]
    if case["call"] == "plan":
        # profiles of three tiers, fastest first, of which the fastest can always meet the objective
        a = [(1_000, 4_000), (4_000, 12_000), (12_000, 20_000)]
        c = [(200, 600), (600, 1_500), (1_500, 3_000)]
        return affine_tables(rng, S, H, B, a, c, jitter=0.05)
    if case["pipeline"] == "tree6":      # CPU-like and accelerator-like hardware
        a, c = [(1_000, 5_000)] + [(8_000, 20_000)] * (H - 1), [(1_500, 3_000)] + [(200, 600)] * (H - 1)
        return affine_tables(rng, S, H, B, a, c)
    return affine_tables(rng, S, H, B, (1_000, 20_000), (200, 3_000), jitter=0.05 if B <= 33 else 0.0)


def _candidates(case, rng):
    S, H, B, R, C = case["stages"], case["hw"], case["max_batch"], case["replicas"], case["candidates"]
    batches = np.array([b for b in (1, 2, 4, 8, 16, 32, 64) if b <= B], np.uint8)
    if case["space"] == "product":
        return product_candidates(rng, S, H, batches, R, [int(k) for k in case["choices"].split(",")])
    cfg = uniform_candidates(rng, C, S, H, batches, R)
    if case["space"] == "step":          # one model of one plan re-chosen per candidate
        plan = np.zeros((S, 4), np.uint8)
        plan[:] = (0, batches[len(batches) // 2], max(2, R // 2), 0)
        model = np.arange(C) % S
        again = cfg[np.arange(C), model]
        cfg[:] = plan
        cfg[np.arange(C), model] = again
    return cfg


class _State:
    pass


def prepare(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    st = _State()
    st.case = case
    parent, bit, val, parent2, probs = _pipe(case)
    S, n = case["stages"], case["queries"]
    lat = _tables(case, rng)
    if case["cv"] > 0.0:
        arrival = gamma_arrivals(rng, n, case["qps"], case["cv"])
    else:                                # the rate ramps up by two thirds over the trace
        arrival = ramp_arrivals(rng, n, case["qps"], case["qps"] / 0.6, n / (case["qps"] / 0.75))
    join = None if parent2 is None else (np.array(parent2, np.int32), np.full(S, -1, np.int8), np.zeros(S, np.uint8))
    st.est = il.Estimator(np.array(parent, np.int32), np.array(bit, np.int8), np.array(val, np.uint8), lat, arrival,
                          bernoulli_bits(rng, n, probs), join=join)
    st.cfg = _candidates(case, rng)
    if case["call"] == "plan":
        st.lat, st.parent, st.prices = lat, np.array(parent), np.array([0.90, 0.35, 0.10])
    elif case["call"] == "envelope":
        st.windows = envelope_windows(int(lat[:, 0, 0].sum()))
    elif case["call"] in ("estimate", "feasible") and case["entry"] == "device":
        st.est.reserve_workspace(len(st.cfg))
        st.cfg = torch.from_numpy(st.cfg).cuda()
    return st


def run(st):
    case, est = st.case, st.est
    slo, on_device = case["slo_us"], case["entry"] == "device"
    if case["call"] == "estimate":
        p99, miss = est.estimate_device(st.cfg, slo) if on_device else est.estimate(st.cfg, slo)
        return {"p99_us": p99, "miss": miss}
    if case["call"] == "feasible":
        return est.feasible_device(st.cfg, slo) if on_device else est.feasible(st.cfg, slo).astype(np.uint8)
    if case["call"] == "latencies":
        return est.latencies(st.cfg[0])
    if case["call"] == "envelope":
        return est.traffic_envelope(st.windows)
    planner = Planner(st.parent, st.lat, est.visits, st.prices, slo, lambda c: est.estimate(c, slo),
                      feasible=lambda c: est.feasible(c, slo))
    plan = planner.minimize_cost()
    return {"feasible": int(plan.feasible), "p99_us": plan.p99_us, "trajectory": np.stack(plan.trajectory) if plan.trajectory
            else np.zeros((0, case["stages"], 4), np.uint8)}


def work(case):
    """What the answer cannot do without.  Bytes: trace, candidates and answers, once each.  Operations: per query
    served at a stage an arrival compared with the dispatch time, counted into its batch, given its finish time and
    passed on (6), and per query that leaves a latency and its comparison (3); a sweep serves a query once per distinct
    chain of choices above and at a stage.  A Planner run counts as 64 candidates."""
    S, n, C = case["stages"], case["queries"], case["candidates"]
    if case["call"] == "envelope":
        W = len(envelope_windows(40_000))
        return {"bytes": 8.0 * n + 16.0 * W, "flops": 2.0 * n * W}
    share = _visits(case)
    if case["space"] == "product":
        k, parent = [int(x) for x in case["choices"].split(",")], _pipe(case)[0]
        nodes = [k[0]]
        for s in range(1, S):
            nodes.append(nodes[parent[s]] * k[s])
        events = sum(m * v for m, v in zip(nodes, share)) * n
    elif case["space"] == "step" and case["call"] != "plan":
        # a stage is only served anew where it or a stage above it was re-chosen
        events = C * n * sum(share) / 2
    else:
        events = (64 if case["call"] == "plan" else C) * n * sum(share)
    answers = 8.0 * n if case["call"] == "latencies" else C * (1.0 if case["call"] == "feasible" else 16.0)
    return {"bytes": 9.0 * n + 4.0 * S * C + answers, "flops": 6.0 * events + 3.0 * n * (1 if case["space"] == "product" else C)}


def tolerance(case):
    return "exact"        # whole microseconds and counts: the simulation is deterministic
