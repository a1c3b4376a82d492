"""The dot-product kernel on instances that no other product kernel takes
(negative entries, nonzero diagonals) above 32 locations: calls in parts, in
every sequential mode, resumed, resumed by and from the table kernels, and in
serving slices. Every replica compared equals the CPU oracle's bit for bit."""

import numpy as np
import pytest

import oracle as O
from gpu_common import check, device, host, library
from paper_2605_24408_gb300 import instances as G

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def signed(n, seed=0, top=127):
    return (G.random_symmetric(n, -60, 70, seed=n + seed, tag=3, diag=True),
            G.random_symmetric(n, -top, top, seed=n + seed, tag=4, diag=True))


def schedule(D, F, kind, S):
    return O.beta_schedule(kind, S, O.beta_max(D, F))


def slots(p, q):
    shape = p.pdit_launch_shape(q, 1 << 20)
    assert shape["influence"] == "products"
    return shape["ctas"] * shape["replicas_per_cta"]


@pytest.mark.parametrize("n,wpr", [(60, 1), (100, 1), (112, 1), (112, 2), (128, 4), (200, 8)])
def test_mappings(n, wpr):
    p = library()
    D, F = signed(n)
    S, R = 6, 7
    beta = schedule(D, F, "geometric", S)
    with p.Qap(D, F) as q:
        p.pdit_set_influence(q, p.PDIT_INFLUENCE_PRODUCTS)
        p.pdit_set_warps_per_replica(q, wpr)
        shape = p.pdit_launch_shape(q, R)
        assert shape["influence"] == "products" and shape["warps_per_replica"] == wpr
        g = host(p.anneal_device(q, R, device(beta), S, 5, per_replica=True))
    check(g, O.anneal(D, F, beta, S, 5, 0, R, threads=7))


@pytest.mark.parametrize("n,S,kind", [(40, 40, "linear"), (100, 24, "geometric"), (112, 16, "linear"),
                                      (140, 16, "geometric")])
def test_parts(n, S, kind):
    p = library()
    D, F = signed(n, 1)
    beta = schedule(D, F, kind, S)
    with p.Qap(D, F) as q:
        R = slots(p, q) + 37
        g = host(p.anneal_device(q, R, device(beta), S, 5, per_replica=True))
    for lo, hi in [(0, 3), (R - 40, R - 37), (R - 3, R)]:
        check(g, O.anneal(D, F, beta, S, 5, lo, hi, threads=3), slice(lo, hi))


def test_parts_resumed_and_fixed():
    """A call too short for parts, then one in parts; fixed betas in parts."""
    p = library()
    D, F = signed(48)
    S = 40
    beta = schedule(D, F, "linear", S)
    bm = O.beta_max(D, F)
    with p.Qap(D, F) as q:
        R = slots(p, q) + 5
        a = p.anneal_device(q, R, device(beta), S, 9, per_replica=True, sweep_end=6)
        g = host(p.anneal_device(q, R, device(beta), S, 9, per_replica=True, sweep_begin=6, resume=True,
                                 workspace=a["workspace"]))
        fb = np.array([bm * (0.2 + 0.01 * (i % 50)) for i in range(R)], np.float32)
        gf = host(p.anneal_device(q, R, device(fb), 16, 4, per_replica=True, mode=p.PDIT_MODE_FIXED))
    for lo, hi in [(0, 2), (R - 2, R)]:
        check(g, O.anneal(D, F, beta, S, 9, lo, hi, threads=2), slice(lo, hi))
        check(gf, O.anneal(D, F, fb[lo:hi], 16, 4, lo, hi, threads=2, mode="fixed"), slice(lo, hi))


def test_tempering_in_parts():
    p = library()
    D, F = signed(40, 2)
    L, S = 5, 13
    ladder = O.beta_schedule("geometric", L, O.beta_max(D, F))
    with p.Qap(D, F) as q:
        R = -(-(slots(p, q) + 37) // L) * L
        g = host(p.anneal_device(q, R, device(ladder), S, 3, per_replica=True, mode=p.PDIT_MODE_PT, ladder_len=L,
                                 exchange_period=4, timeout_periods=2))
    for lo, hi in [(0, L), (R - L, R)]:
        r = O.anneal(D, F, ladder, S, 3, lo, hi, threads=L, mode="pt", ladder_len=L, period=4, timeout=2)
        check(g, r, slice(lo, hi))
        assert np.array_equal(g["replica_rung"][lo:hi], r["rung"])


@pytest.mark.parametrize("n,S,cut", [(100, 30, 13), (90, 24, 10)])
def test_resumed_across_kernels(n, S, cut):
    p = library()
    D, F = signed(n, 3)
    beta = schedule(D, F, "linear", S)
    R = 12
    r = O.anneal(D, F, beta, S, 6, 0, R, threads=8)
    pr, tb = p.PDIT_INFLUENCE_PRODUCTS, p.PDIT_INFLUENCE_TABLE
    for first, second in ((pr, pr), (pr, tb), (tb, pr)):
        with p.Qap(D, F) as q:
            p.pdit_set_influence(q, first)
            a = p.anneal_device(q, R, device(beta), S, 6, per_replica=True, sweep_end=cut)
            p.pdit_set_influence(q, second)
            g = host(p.anneal_device(q, R, device(beta), S, 6, per_replica=True, sweep_begin=cut, resume=True,
                                     workspace=a["workspace"]))
        check(g, r)


def test_tempering_resumed_across_kernels():
    """The permuted flow matrices kept between exchange periods, rebuilt by a
    resumed call."""
    p = library()
    D, F = signed(64)
    ladder = O.beta_schedule("geometric", 4, O.beta_max(D, F))
    R, S, cut = 12, 26, 10
    r = O.anneal(D, F, ladder, S, 8, 0, R, threads=R, mode="pt", ladder_len=4, period=3, timeout=2)
    kw = dict(mode=p.PDIT_MODE_PT, ladder_len=4, exchange_period=3, timeout_periods=2, per_replica=True)
    pr, tb = p.PDIT_INFLUENCE_PRODUCTS, p.PDIT_INFLUENCE_TABLE
    for first, second in ((pr, tb), (tb, pr), (pr, pr)):
        with p.Qap(D, F) as q:
            ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")  # room for either kernel
            p.pdit_set_influence(q, first)
            p.anneal_device(q, R, device(ladder), S, 8, sweep_end=cut, workspace=ws, **kw)
            p.pdit_set_influence(q, second)
            g = host(p.anneal_device(q, R, device(ladder), S, 8, sweep_begin=cut, resume=True, workspace=ws, **kw))
        check(g, r)
        assert np.array_equal(g["replica_rung"], r["rung"])


def test_serving_slices():
    """Dot-product requests and table-only ones (entries beyond a byte, some
    negative), in many short slices."""
    p = library()
    S, R = 70, 16
    insts = [signed(50), signed(100), signed(24), signed(40, 5, top=300), signed(70, 6, top=300)]
    srv = p.Server(slice_sweeps=7, max_active=8)
    tickets = [srv.submit(D, F, R, S, 2, k) for k, (D, F) in enumerate(insts)]
    while sum(srv.tick()):
        pass
    for k, (D, F) in enumerate(insts):
        state, perm, cost, _ = srv.result(tickets[k])
        r = O.anneal(D, F, schedule(D, F, "linear", S), S, 2, 0, R, inst=k, threads=8)
        assert state == 2 and cost == r["cost"] and np.array_equal(perm, r["perm"])
    srv.close()
