"""Calls with few replicas an SM, where the automatic choice takes a kernel
that puts several warps on a replica instead of the tensor-core product
kernel: which one runs on each side of the lines, and that replicas equal the
CPU oracle's there; and the product kernel at those sizes when one warp per
replica is asked for."""

import numpy as np
import pytest

import oracle as O
from gpu_common import check, device, host, library, sms
from paper_2605_24408_gb300 import instances as G

pytestmark = pytest.mark.gpu


def compare(p, q, D, F, beta, S, R, mode="anneal", L=4):
    kw, okw, step = {}, {}, 1
    if mode == "pt":
        kw = dict(mode=p.PDIT_MODE_PT, ladder_len=L, exchange_period=2, timeout_periods=2)
        okw, step = dict(mode="pt", ladder_len=L, period=2, timeout=2), L
    g = host(p.anneal_device(q, R, device(beta), S, 6, per_replica=True, **kw))
    for lo in {0, (R - 1) // step * step - step * (3 if step == 1 else 0)}:
        lo = max(0, lo)
        hi = min(R, lo + 4)
        r = O.anneal(D, F, beta, S, 6, lo, hi, threads=4, **okw)
        check(g, r, slice(lo, hi))


@pytest.mark.parametrize("n,per_sm,warps", [(112, 1, 1), (113, 2, 2), (128, 2, 2), (128, 3, 1), (129, 1, 1), (160, 2, 4),
                                            (160, 3, 1), (192, 2, 4), (192, 3, 1), (200, 3, 4), (200, 4, 1), (224, 2, 8),
                                            (224, 3, 1),
                                            (225, 1, 8), (225, 2, 1), (256, 1, 8)])
def test_symmetric(n, per_sm, warps):
    """`warps` at per_sm replicas an SM: 1 is the product kernel (the first
    call that fills the SM to per_sm), more the dot-product kernel (the last)."""
    p = library()
    D, F = G.dense_instance(n, seed=n)
    S = 3
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    R = sms() * per_sm if warps > 1 else sms() * (per_sm - 1) + 1
    for infl in (p.PDIT_INFLUENCE_AUTO, p.PDIT_INFLUENCE_PRODUCTS):
        with p.Qap(D, F) as q:
            p.pdit_set_influence(q, infl)
            shape = p.pdit_launch_shape(q, R)
            assert shape["influence"] == "products" and shape["warps_per_replica"] == warps
            compare(p, q, D, F, beta, S, R)


@pytest.mark.parametrize("n,per_sm,dot", [(120, 1, False), (176, 1, True), (176, 2, False), (200, 2, True),
                                          (200, 3, False), (224, 2, True), (240, 1, True), (240, 2, False)])
def test_symmetric_tempering(n, per_sm, dot):
    p = library()
    D, F = G.dense_instance(n, seed=n + 1)
    L, S = 4, 5
    beta = O.beta_schedule("geometric", L, O.beta_max(D, F))
    R = (sms() * per_sm if dot else sms() * (per_sm - 1) + L) // L * L
    with p.Qap(D, F) as q:
        # the dot-product kernel's permuted matrices are kept between exchange periods
        o = p.opts(replicas=R, sweeps=S, mode=p.PDIT_MODE_PT, ladder_len=L)
        assert (p.pdit_workspace_bytes(q, o) > R * n * n) == dot
        compare(p, q, D, F, beta, S, R, "pt", L)


def general(n):
    return G.asymmetric(n, 0, 99, n, 101), G.asymmetric(n, 0, 99, n, 103)


@pytest.mark.parametrize("n,per_sm,kind", [(50, 1, "products"), (75, 1, "products"), (79, 5, "table"),
                                           (100, 5, "table"), (100, 6, "products"), (112, 3, "table"),
                                           (112, 4, "products"), (113, 2, "table"), (128, 2, "table"),
                                           (128, 3, "products"), (129, 2, "table"), (144, 3, "products"),
                                           (160, 1, "table"), (160, 2, "products")])
def test_general(n, per_sm, kind):
    """The last call of the table kernels, the first of the product kernel."""
    p = library()
    D, F = general(n)
    S = 3
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    R = sms() * per_sm if kind == "table" else max(8, sms() * (per_sm - 1) + 1)
    with p.Qap(D, F) as q:
        assert p.pdit_launch_shape(q, R)["influence"] == kind
        compare(p, q, D, F, beta, S, R)


@pytest.mark.parametrize("n,per_sm,tables", [(75, 1, False), (100, 2, True), (100, 3, False), (120, 1, False),
                                             (144, 2, True), (160, 1, True), (160, 2, False)])
def test_general_tempering(n, per_sm, tables):
    p = library()
    D, F = general(n)
    L, S = 4, 5
    beta = O.beta_schedule("geometric", L, O.beta_max(D, F))
    R = (sms() * per_sm if tables else sms() * (per_sm - 1) + 8) // L * L
    with p.Qap(D, F) as q:
        o = p.opts(replicas=R, sweeps=S, mode=p.PDIT_MODE_PT, ladder_len=L)
        assert (p.pdit_workspace_bytes(q, o) > 4 * R * n * n) == tables
        compare(p, q, D, F, beta, S, R, "pt", L)


@pytest.mark.parametrize("n", [113, 128, 129, 160, 161, 192, 193, 224, 225, 256])
def test_product_kernel_with_one_warp_asked(n):
    p = library()
    D, F = G.dense_instance(n, seed=n)
    S = 4
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    with p.Qap(D, F) as q:
        p.pdit_set_warps_per_replica(q, 1)
        # (its shared memory does not depend on the replicas)
        a, b = p.pdit_launch_shape(q, 1), p.pdit_launch_shape(q, 1 << 16)
        assert a["influence"] == "products" and a["smem_bytes"] == b["smem_bytes"]
        compare(p, q, D, F, beta, S, 5)


def instance(kind, n):
    if kind == "general":
        return general(n)
    if kind == "wide":
        return G.dense_symmetric(n, 0, 999, n, tag=23), G.dense_symmetric(n, 0, 999, n, tag=33)
    return G.dense_instance(n, seed=n)


MULTI = [("general", 76), ("general", 100), ("general", 128), ("general", 160), ("wide", 112), ("dense", 176),
         ("dense", 200), ("dense", 224), ("dense", 256)]


@pytest.mark.parametrize("kind,n", MULTI)
def test_batches(kind, n):
    """Few replicas in all: the kernels of a single call, spread over the SMs
    (a shape class that one warp per replica does not share), and the results
    of the oracle; many: the product kernel."""
    p = library()
    few = kind != "wide" and n > 76
    D, F = instance(kind, n)
    S = 2
    qs = [p.Qap(D, F), p.Qap(D, F)]
    p.pdit_set_warps_per_replica(qs[1], 1)  # the product kernel
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    for R, classes in ((20, 2 if few else 1), (4 * sms(), 1)):
        items = [{"qap": q, "replicas": R, "sweeps": S, "beta": device(beta), "seed": 4, "instance_id": k}
                 for k, q in enumerate(qs)]
        batch = p.Batch(items)
        assert batch.info()[0] == classes
        if R == 20:
            batch.run()
            for k, o in enumerate([host(o) for o in batch.out]):
                r = O.anneal(D, F, beta, S, 4, 0, R, inst=k, threads=8)
                assert int(o["best_cost"][0]) == r["cost"] and np.array_equal(o["best_perm"], r["perm"])
        batch.close()
    for q in qs:
        q.close()


def test_served():
    """Few served replicas: slices on the kernels that batches take."""
    p = library()
    S, R = 9, 10
    srv = p.Server(slice_sweeps=4, max_active=16)
    insts = [instance(kind, n) for kind, n in MULTI]
    tickets = [srv.submit(D, F, R, S, 5, k) for k, (D, F) in enumerate(insts)]
    while sum(srv.tick()):
        pass
    for k, (D, F) in enumerate(insts):
        state, perm, cost, _ = srv.result(tickets[k])
        r = O.anneal(D, F, O.beta_schedule("linear", S, O.beta_max(D, F)), S, 5, 0, R, inst=k, threads=8)
        assert state == 2 and cost == r["cost"] and np.array_equal(perm, r["perm"])
    srv.close()


@pytest.mark.parametrize("n,R", [(120, 5), (128, 8)])
def test_batch_units_of_one_round(n, R):
    """Loads where units of 4 replicas would no longer fit the SMs at once:
    the batch equals single calls."""
    p = library()
    D, F = general(n)
    R *= sms()
    S = 2
    with p.Qap(D, F) as q:
        db = device(O.beta_schedule("linear", S, O.beta_max(D, F)))
        items = [{"qap": q, "replicas": R // 2 + k, "sweeps": S, "beta": db, "seed": 4, "instance_id": k}
                 for k in range(2)]
        batch = p.Batch(items)
        batch.run()
        for k, o in enumerate([host(o) for o in batch.out]):
            g = host(p.anneal_device(q, R // 2 + k, db, S, 4, instance_id=k))
            assert int(o["best_cost"][0]) == int(g["best_cost"][0]) and np.array_equal(o["best_perm"], g["best_perm"])
        batch.close()
