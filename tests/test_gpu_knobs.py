"""A table knob gets the table kernels, also where the automatic choice keeps
no table: every setting that asks for them, at sizes of the small kernel, the
product kernel and its wide and general forms. Tempering keeps every replica's
table in the workspace, which tells the kernels apart."""

import numpy as np
import pytest

import oracle as O
from gpu_common import check, device, host, library
from paper_2605_24408_gb300 import instances as G

pytestmark = pytest.mark.gpu

INSTANCES = {"small": lambda: G.dense_instance(30, seed=4), "smallest": lambda: G.dense_instance(12, seed=4),
             "products": lambda: G.dense_instance(75, seed=4),
             "wide": lambda: (G.dense_symmetric(61, 0, 999, 1, tag=23), G.dense_symmetric(61, 0, 999, 1, tag=33)),
             "general": lambda: (G.asymmetric(50, 0, 99, 1, 101), G.asymmetric(50, 0, 99, 1, 103))}


@pytest.mark.parametrize("which", list(INSTANCES))
@pytest.mark.parametrize("knob", [None, "influence", "pending", "placement"])
def test_table_knobs(which, knob):
    p = library()
    D, F = INSTANCES[which]()
    n, R, S = len(D), 12, 8
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    with p.Qap(D, F) as q:
        p.pdit_set_class_update(q, False)
        if knob == "influence":
            p.pdit_set_influence(q, p.PDIT_INFLUENCE_TABLE)
        elif knob == "pending":
            p.pdit_set_pending_swaps(q, 1)
        elif knob == "placement":
            p.pdit_set_table_placement(q, p.PDIT_PLACE_SHARED)
        o = p.opts(replicas=R, sweeps=S, mode=p.PDIT_MODE_PT, ladder_len=R)
        assert (p.pdit_workspace_bytes(q, o) > 4 * R * n * n) == (knob is not None)
        g = host(p.anneal_device(q, R, device(beta), S, 2, per_replica=True))
    check(g, O.anneal(D, F, beta, S, 2, 0, R, threads=8))


def test_autotuned_small_instance():
    """The tuner times the tables themselves beside the built-in choice, and
    leaves a handle that runs one of them."""
    p = library()
    D, F = G.dense_instance(24, seed=9)
    R, S = 40, 12
    beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
    with p.Qap(D, F) as q:
        p.pdit_autotune(q, R, device(beta), S)
        g = host(p.anneal_device(q, R, device(beta), S, 7, per_replica=True))
    check(g, O.anneal(D, F, beta, S, 7, 0, R, threads=8))
