"""The work this framework is used for, as measurable cases.

Every case is a whole solve (or a bounded slice of one: fewer sweeps of the
same schedule) through the public entry points of
`paper_2605_24408_gb300.pdit`: the host-buffer call, the device-buffer call in
each mode, the graph-captured batch and the serving loop. Sizes are those of
the named workloads of `instances.py`, of `bench.py` and of the tests; the
schedules are the library's own. All outputs are whole numbers (permutations,
costs, counts, status bits), a pure function of the instance, the schedule and
the sampler's seed.
"""

from __future__ import annotations

import numpy as np
import torch

from paper_2605_24408_gb300 import instances as G
from paper_2605_24408_gb300 import pdit as P

# Arithmetic of one candidate of one p-dit update that no implementation
# avoids: the swap energy of Eq. 3 from its influence entries (7), the shift
# and scale of the Boltzmann weight (2), the exponential (a range reduction of
# 4 and a degree-7 polynomial of 14) and the running sum (1). Keeping the
# influence entries current comes on top and depends on the acceptance rate.
OPS_PER_CANDIDATE = 28


def listed():
    return [
        # The smallest workload of the paper's shape (3 x 4 grid, 64 replicas,
        # the full 1000-sweep schedule) as a script runs it: host matrices in,
        # create, solve, destroy. Latency of one update chain.
        {"name": "host_n12", "call": "host", "inst": "grid", "n": 12, "replicas": 64, "sweeps": 1000,
         "schedule": "linear"},
        # The 5 x 6 grid workload, complete: 1024 replicas, 5000 geometric sweeps.
        {"name": "grid_n30", "call": "anneal", "inst": "grid", "n": 30, "replicas": 1024, "sweeps": 5000,
         "schedule": "geometric"},
        # An ordinary mid-size solve of a grid instance at an odd size, with
        # few replicas: a GPU that is not filled.
        {"name": "grid_n75", "call": "anneal", "inst": "grid", "n": 75, "replicas": 300, "sweeps": 400,
         "schedule": "linear"},
        # The headline workload (dense N = 100, 4096 replicas), a twentieth
        # of its sweeps over the same range of beta.
        {"name": "dense_n100", "call": "anneal", "inst": "dense", "n": 100, "replicas": 4096, "sweeps": 500,
         "schedule": "linear"},
        # The largest size: dense N = 256.
        {"name": "dense_n256", "call": "anneal", "inst": "dense", "n": 256, "replicas": 2048, "sweeps": 60,
         "schedule": "linear"},
        # Entries beyond a byte (values to 999 in D and F), an odd size.
        {"name": "wide_n61", "call": "anneal", "inst": "wide", "n": 61, "replicas": 512, "sweeps": 500,
         "schedule": "geometric"},
        # The general QAP (neither matrix symmetric), N = 100.
        {"name": "general_n100", "call": "anneal", "inst": "general", "n": 100, "replicas": 4096, "sweeps": 150,
         "schedule": "linear"},
        # Two-level flow at the size of tai256c (92 of 256 facilities).
        {"name": "classes_n256", "call": "anneal", "inst": "classes", "n": 256, "replicas": 4096, "sweeps": 150,
         "schedule": "linear"},
        # Parallel tempering: 409 ladders of 10 rungs, exchanges every 4 sweeps.
        {"name": "tempering_n100", "call": "tempering", "inst": "dense", "n": 100, "replicas": 4090, "sweeps": 100,
         "schedule": "geometric"},
        # Concurrent updates (the GPU-CUPIM variant).
        {"name": "concurrent_n100", "call": "concurrent", "inst": "dense", "n": 100, "replicas": 4096,
         "sweeps": 100, "schedule": "linear"},
        # A ragged batch, N uniform in 12..256, grid and dense instances in
        # turn, replayed as a captured graph.
        {"name": "batch_ragged", "call": "batch", "inst": "ragged", "n": 256, "count": 24, "replicas": 256,
         "sweeps": 100, "schedule": "linear"},
        # A burst of serving requests, N uniform in 20..200, in slices of 50 sweeps.
        {"name": "served_burst", "call": "serve", "inst": "ragged", "n": 200, "count": 16, "replicas": 512,
         "sweeps": 100, "schedule": "linear"},
    ]


# Upper bound of a drawn case: replicas x sweeps x n^2 (candidates visited) of
# dense_n256, which takes the longest per candidate among the listed cases
# near that count.
MAX_CANDIDATES = 2048 * 60 * 256 * 256


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    call = rng.choice(["host", "anneal", "anneal", "anneal", "anneal", "tempering", "concurrent", "batch", "serve"])
    inst = rng.choice(["grid", "dense", "dense", "wide", "general", "classes"])
    c = {"call": call, "schedule": rng.choice(["linear", "geometric"])}
    if call in ("batch", "serve"):
        c["inst"] = "ragged"
        c["n"] = rng.randint(60, 256) if call == "batch" else rng.randint(60, 200)
        c["count"] = rng.randint(4, 24)
        c["replicas"] = _log_int(rng, 64, 512)
        cand = c["count"] * c["replicas"] * c["n"] ** 2
    else:
        # wide values stay below the library's int32 range check up to n = 120
        c["inst"] = inst
        c["n"] = _log_int(rng, 12, 120 if inst == "wide" else 256)
        c["replicas"] = _log_int(rng, 64, 4096)
        if call == "tempering":
            c["replicas"] = max(10, c["replicas"] // 10 * 10)
        cand = c["replicas"] * c["n"] ** 2
    c["sweeps"] = _log_int(rng, 10, max(11, min(1000, MAX_CANDIDATES // (2 * cand))))
    return c


def _instance(inst, n, seed):
    if inst == "grid":
        rows, cols = (3, 4) if n == 12 else (5, 6) if n == 30 else G.near_square_grid(n)
        return G.grid_instance(rows, cols, 0.5 if n == 12 else 0.4, seed, n)
    if inst == "dense":
        return G.dense_instance(n, seed)
    if inst == "wide":
        return G.dense_symmetric(n, 0, 999, seed, tag=23), G.dense_symmetric(n, 0, 999, seed, tag=33)
    if inst == "general":
        return G.asymmetric(n, 0, 99, seed, 101), G.asymmetric(n, 0, 99, seed, 103)
    if inst == "classes":
        return G.flow_class_instance(n, max(1, n * 92 // 256), seed)
    raise KeyError(inst)


def _sizes(case):
    """Sizes of a batch or of a burst of requests: uniform over the range, the
    largest always among them; by position, so that every seed has the same
    amount of work."""
    lo = 12 if case["call"] == "batch" else 20
    return [case["n"] if k == 0 else G.ragged_size(k, 5, lo, case["n"]) for k in range(case["count"])]


def _ragged(case, seed):
    return [G.ragged_instance(k, n, seed) for k, n in enumerate(_sizes(case))]


def prepare(case, seed):
    S = case["sweeps"]
    st = {"case": case, "seed": seed}
    if case["call"] == "batch":
        items = []
        for k, (D, F) in enumerate(_ragged(case, seed)):
            q = P.Qap(D, F)
            beta = P.pdit_beta_schedule(case["schedule"], S, P.pdit_beta_max(q))
            items.append({"qap": q, "replicas": case["replicas"], "sweeps": S, "beta": torch.from_numpy(beta).cuda(),
                          "seed": seed, "instance_id": k})
        st["stream"] = torch.cuda.Stream()
        st["batch"] = P.Batch(items, graph=True)
        return st
    if case["call"] == "serve":
        st["requests"] = []
        for D, F in _ragged(case, seed):
            with P.Qap(D, F) as q:
                beta = P.pdit_beta_schedule(case["schedule"], S, P.pdit_beta_max(q))
            st["requests"].append((D, F, beta))
        st["server"] = P.Server(slice_sweeps=50, max_active=64)
        return st
    D, F = _instance(case["inst"], case["n"], seed)
    q = P.Qap(D, F)
    bmax = P.pdit_beta_max(q)
    if case["call"] == "host":
        st["D"], st["F"] = D, F
        st["beta"] = P.pdit_beta_schedule(case["schedule"], S, bmax)
        q.close()
        return st
    st["qap"] = q
    if case["call"] == "tempering":
        beta = P.pdit_beta_ladder(bmax / 100.0, bmax, 10)
    else:
        beta = P.pdit_beta_schedule(case["schedule"], S, bmax)
    st["beta"] = torch.from_numpy(np.ascontiguousarray(beta)).cuda()
    return st


def run(state):
    c, seed = state["case"], state["seed"]
    if c["call"] == "host":
        q = P.qap_create(state["D"], state["F"])
        perm, cost = P.pdit_anneal(q, c["replicas"], state["beta"], c["sweeps"], seed)
        P.qap_destroy(q)
        return perm, cost
    if c["call"] == "batch":
        st = state["stream"]
        st.wait_stream(torch.cuda.current_stream())
        state["batch"].run(st)
        torch.cuda.current_stream().wait_stream(st)
        return [(o["best_perm"], o["best_cost"]) for o in state["batch"].out]
    if c["call"] == "serve":
        srv = state["server"]
        tickets = [srv.submit(D, F, c["replicas"], c["sweeps"], seed, rid, beta)
                   for rid, (D, F, beta) in enumerate(state["requests"])]
        while True:
            active, queued = srv.tick()
            if active + queued == 0:
                break
        got = [srv.result(t) for t in tickets]
        return [(state_, perm, cost) for state_, perm, cost, _latency in got]
    kw = {}
    if c["call"] == "tempering":
        kw = {"mode": P.PDIT_MODE_PT, "ladder_len": 10, "exchange_period": 4, "timeout_periods": 100}
    elif c["call"] == "concurrent":
        kw = {"mode": P.PDIT_MODE_CUPIM}
    out = P.anneal_device(state["qap"], c["replicas"], state["beta"], c["sweeps"], seed, per_replica=True, **kw)
    return {k: v for k, v in out.items() if k != "workspace"}


def work(case):
    """What one pass cannot do without: the matrices and the schedule in, the
    results out, and the arithmetic of every candidate of every update."""
    S, R = case["sweeps"], case["replicas"]
    if case["call"] in ("batch", "serve"):
        ns = _sizes(case)
        return {"bytes": sum(8 * n * n + 4 * S + 4 * n + 8 for n in ns),
                "flops": sum(float(OPS_PER_CANDIDATE) * R * S * n * n for n in ns)}
    n = case["n"]
    if case["call"] == "host":
        nbytes = 8 * n * n + 4 * S + 4 * n + 8
    else:
        nbytes = 8 * n * n + 4 * S + 4 * n + 12 + R * (8 * n + 28)
    return {"bytes": nbytes, "flops": float(OPS_PER_CANDIDATE) * R * S * n * n}


def exact(case, seed):
    """Every output is a whole number that the sampler's draws decide; none
    has a value in another arithmetic, so all are compared as they are."""
    return None
