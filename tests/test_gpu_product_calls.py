"""The tensor-core product kernel in calls that its size tests do not make:
parts in every form and lane count, time to target and stopping (also of the
concurrent kernel and in batches), and the largest sums its accumulators are
relied on for. Every replica compared equals the CPU oracle's bit for bit."""

import numpy as np
import pytest

import oracle as O
from gpu_common import check, device, host, library
from paper_2605_24408_gb300 import instances as G

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def instance(form, n):
    if form == "wide":
        return G.dense_symmetric(n, 0, 999, n, tag=23), G.dense_symmetric(n, 0, 999, n, tag=33)
    if form == "general":
        return G.asymmetric(n, 0, 99, n, 101), G.asymmetric(n, 0, 99, n, 103)
    return G.dense_instance(n, seed=n)


def handle(p, D, F):
    """A handle that runs the product kernel at any replica count."""
    q = p.Qap(D, F)
    p.pdit_set_warps_per_replica(q, 1)
    shape = p.pdit_launch_shape(q, 1 << 20)
    # (its shared memory does not depend on the replicas)
    assert p.pdit_launch_shape(q, 1)["smem_bytes"] == shape["smem_bytes"]
    return q, shape["ctas"] * shape["replicas_per_cta"]


FORMS = [("symmetric", 40), ("symmetric", 100), ("symmetric", 150), ("symmetric", 250), ("general", 50),
         ("general", 100), ("general", 150), ("wide", 61), ("wide", 120)]


@pytest.mark.parametrize("form,n", FORMS)
def test_parts(form, n):
    """More replicas than slots, not a whole number of blocks: sweeps in parts,
    each block resuming from what the part before published."""
    p = library()
    D, F = instance(form, n)
    S = 24 if n < 200 else 16
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    q, slots = handle(p, D, F)
    R = slots + 37
    g = host(p.anneal_device(q, R, device(beta), S, 5, per_replica=True))
    for lo, hi in [(0, 3), (R - 40, R - 37), (R - 3, R)]:
        check(g, O.anneal(D, F, beta, S, 5, lo, hi, threads=3), slice(lo, hi))
    q.close()


@pytest.mark.parametrize("form,n", [("symmetric", 40), ("general", 50), ("wide", 61), ("symmetric", 150)])
def test_parts_resumed_tempered_and_fixed(form, n):
    p = library()
    D, F = instance(form, n)
    L, S = 5, 20
    bm = O.beta_max(D, F)
    beta, ladder = O.beta_schedule("linear", S, bm), O.beta_schedule("geometric", L, bm)
    q, slots = handle(p, D, F)
    R = -(-(slots + 37) // L) * L
    a = p.anneal_device(q, R, device(beta), S, 9, per_replica=True, sweep_end=3)
    g = host(p.anneal_device(q, R, device(beta), S, 9, per_replica=True, sweep_begin=3, resume=True,
                             workspace=a["workspace"]))
    t = host(p.anneal_device(q, R, device(ladder), 9, 3, per_replica=True, mode=p.PDIT_MODE_PT, ladder_len=L,
                             exchange_period=4, timeout_periods=2))
    fb = np.array([bm * (0.2 + 0.01 * (i % 50)) for i in range(R)], np.float32)
    f = host(p.anneal_device(q, R, device(fb), 16, 4, per_replica=True, mode=p.PDIT_MODE_FIXED))
    for lo, hi in [(0, L), (R - L, R)]:
        check(g, O.anneal(D, F, beta, S, 9, lo, hi, threads=L), slice(lo, hi))
        r = O.anneal(D, F, ladder, 9, 3, lo, hi, threads=L, mode="pt", ladder_len=L, period=4, timeout=2)
        check(t, r, slice(lo, hi))
        assert np.array_equal(t["replica_rung"][lo:hi], r["rung"])
        check(f, O.anneal(D, F, fb[lo:hi], 16, 4, lo, hi, threads=L, mode="fixed"), slice(lo, hi))
    q.close()


def eq1(D, F, perm):
    return int((D.astype(np.int64) * F[np.ix_(perm, perm)]).sum())


def stopped(g, D, F, target, S):
    """What a stopped call promises: some replica reached the target, and every
    replica's state is whole."""
    assert int(g["status"][0]) == 0
    assert int(g["best_cost"][0]) <= target and -1 <= int(g["reach_sweep"][0]) < S
    for k in range(0, len(g["replica_final_cost"]), max(1, len(g["replica_final_cost"]) // 40)):
        perm = g["replica_final_perm"][k]
        assert np.array_equal(np.sort(perm), np.arange(len(D)))
        assert eq1(D, F, perm) == int(g["replica_final_cost"][k])
        assert eq1(D, F, g["replica_best_perm"][k]) == int(g["replica_best_cost"][k])


@pytest.mark.parametrize("form,n,mode", [("symmetric", 48, "anneal"), ("symmetric", 150, "anneal"),
                                         ("general", 50, "anneal"), ("wide", 61, "anneal"),
                                         ("symmetric", 48, "cupim"), ("symmetric", 100, "cupim")])
def test_target_and_stop(form, n, mode):
    p = library()
    D, F = instance(form, n)
    S, R = 30, 20
    beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
    kw = {"mode": p.PDIT_MODE_CUPIM} if mode == "cupim" else {}
    r = O.anneal(D, F, beta, S, 1, 0, R, threads=8, mode=mode)
    target = int(np.sort(r["best_cost"])[R // 2])
    ro = O.anneal(D, F, beta, S, 1, 0, R, threads=8, mode=mode, target=target)
    start = O.anneal(D, F, beta[:0], 0, 1, 0, R)
    if mode == "cupim":
        q, slots = p.Qap(D, F), 4 * torch.cuda.get_device_properties(0).multi_processor_count
    else:
        q, slots = handle(p, D, F)

    def call(R, target, stop):
        t = torch.tensor([target], dtype=torch.int64, device="cuda")
        return host(p.anneal_device(q, R, device(beta), S, 1, per_replica=True, target=t, stop_at_target=stop, **kw))

    g = call(R, target, False)
    check(g, r)
    assert int(g["reach_sweep"][0]) == int(ro["reach_sweep"].min())
    # a target that nothing reaches: the flag is read, nobody stops
    check(call(R, int(r["best_cost"].min()) - 1, True), r)
    # one that every initial state reaches: nobody starts
    g = call(R, int(start["final_cost"].max()), True)
    assert int(g["reach_sweep"][0]) == -1 and not g["replica_accepted"].any()
    assert np.array_equal(g["replica_final_perm"], start["final_perm"])
    stopped(call(R, target, True), D, F, target, S)
    stopped(call(slots + 37, target, True), D, F, target, S)  # in parts
    q.close()


def test_batch_stops_at_target():
    p = library()
    S, R = 40, 40
    items, wants = [], []
    for k, (form, n) in enumerate([("symmetric", 100), ("general", 50), ("wide", 61), ("symmetric", 150)]):
        D, F = instance(form, n)
        q, _ = handle(p, D, F)
        beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
        r = O.anneal(D, F, beta, S, 3, 0, R, inst=k, threads=8)
        target = int(np.sort(r["best_cost"])[R // 2])
        wants.append((D, F, target, r))
        items.append({"qap": q, "replicas": R, "sweeps": S, "beta": device(beta), "seed": 3, "instance_id": k,
                      "target": torch.tensor([target], dtype=torch.int64, device="cuda")})
    for stop in (False, True):
        batch = p.Batch(items, stop_at_target=stop)
        batch.run()
        for o, (D, F, target, r) in zip([host(o) for o in batch.out], wants):
            assert eq1(D, F, o["best_perm"]) == int(o["best_cost"][0]) <= target
            assert 0 <= int(o["reach_sweep"][0]) < S
            if not stop:
                assert int(o["best_cost"][0]) == r["cost"] and np.array_equal(o["best_perm"], r["perm"])
        batch.close()
    for it in items:
        it["qap"].close()


@pytest.mark.parametrize("form,n,dlo,dhi,flo,fhi", [("symmetric", 256, 126, 127, 126, 127),
                                                    ("symmetric", 128, 126, 127, 126, 127),
                                                    ("wide", 128, 2040, 2047, 490, 503),
                                                    ("wide", 128, 490, 503, 2040, 2047),
                                                    ("general", 128, 126, 127, 126, 127),
                                                    ("cupim", 112, 126, 127, 126, 127), ("cupim", 128, 126, 127, 126, 127)])
def test_largest_sums(form, n, dlo, dhi, flo, fhi):
    """Entries at the top of their range: sums of products to 8.3e6 units below
    the 2^24 that binary32 holds exactly, in the accumulators too."""
    p = library()
    if form == "general":
        D, F = G.asymmetric(n, dlo, dhi, 1, 101), G.asymmetric(n, flo, fhi, 1, 103)
    else:
        D, F = G.dense_symmetric(n, dlo, dhi, 1, tag=3), G.dense_symmetric(n, flo, fhi, 2, tag=5)
    S, R = 6, 5
    mode = "cupim" if form == "cupim" else "anneal"
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    r = O.anneal(D, F, beta, S, 4, 0, R, threads=5, mode=mode)
    if mode == "cupim":
        q, kw = p.Qap(D, F), {"mode": p.PDIT_MODE_CUPIM}
    else:
        (q, _), kw = handle(p, D, F), {}
    check(host(p.anneal_device(q, R, device(beta), S, 4, per_replica=True, **kw)), r)
    q.close()
