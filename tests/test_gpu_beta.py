"""Betas outside the finite range. The library reads device schedules as they
are, so every kernel has to answer them in bounds: no outcome has a weight
under an infinite beta or a NaN, and every location stays. Sweeps of finite
beta among them run as if the others were not there."""

import numpy as np
import pytest

import oracle as O
from gpu_common import KEYS, device, host, library
from paper_2605_24408_gb300 import instances as G

pytestmark = pytest.mark.gpu


def instance(kind, n):
    if kind == "wide":
        return G.dense_symmetric(n, 0, 999, n, tag=23), G.dense_symmetric(n, 0, 999, n, tag=33)
    if kind == "general":
        return G.asymmetric(n, 0, 99, n, 101), G.asymmetric(n, 0, 99, n, 103)
    if kind == "signed":
        return (G.random_symmetric(n, -60, 70, seed=n, tag=3, diag=True),
                G.random_symmetric(n, -127, 127, seed=n, tag=4, diag=True))
    if kind == "classes":
        return G.flow_class_instance(n, n // 3, n)
    return G.dense_instance(n, seed=n)


# every kernel: products (16 and 32 lanes, general, wide), small, dot products
# with one and more warps, tables, flow classes, concurrent products and tables
CASES = [("dense", 100, 1, None), ("dense", 200, 1, None), ("general", 75, 1, None), ("wide", 61, 1, None),
         ("dense", 30, 0, None), ("signed", 24, 0, None), ("signed", 40, 1, None), ("signed", 77, 2, None),
         ("signed", 140, 4, None), ("dense", 50, 0, "table"), ("dense", 120, 4, "table"), ("classes", 60, 0, None),
         ("dense", 20, 0, "cupim"), ("dense", 100, 0, "cupim"), ("signed", 33, 0, "cupim")]


@pytest.mark.parametrize("kind,n,wpr,how", CASES)
def test_nothing_moves_without_a_weight(kind, n, wpr, how):
    p = library()
    D, F = instance(kind, n)
    bm = O.beta_max(D, F)
    R, seed = 6, 5
    kw = {"mode": p.PDIT_MODE_CUPIM} if how == "cupim" else {}
    start = O.anneal(D, F, np.zeros(0, np.float32), 0, seed, 0, R)
    with p.Qap(D, F) as q:
        if wpr:
            p.pdit_set_warps_per_replica(q, wpr)
        if how == "table":
            p.pdit_set_influence(q, p.PDIT_INFLUENCE_TABLE)
        for bad in (np.inf, np.nan):
            g = host(p.anneal_device(q, R, device(np.full(3, bad)), 3, seed, per_replica=True, **kw))
            assert int(g["status"][0]) == 0
            assert np.array_equal(g["replica_final_perm"], start["final_perm"])
            assert np.array_equal(g["replica_final_cost"], start["final_cost"])
            assert not g["replica_accepted"].any()
        # finite sweeps between: as calls of these sweeps alone
        S = 5
        db = device([bm / 4, np.inf, bm / 2, np.nan, bm])
        g = host(p.anneal_device(q, R, db, S, seed, per_replica=True, **kw))
        a = p.anneal_device(q, R, db, S, seed, per_replica=True, sweep_end=1, **kw)
        for s in (2, 4):
            a = p.anneal_device(q, R, db, S, seed, per_replica=True, sweep_begin=s, sweep_end=s + 1, resume=True,
                                workspace=a["workspace"], **kw)
        a = host(a)
    assert int(g["status"][0]) == 0
    for k in KEYS:
        assert np.array_equal(g["replica_" + k], a["replica_" + k]), k
    assert g["replica_accepted"].all()
