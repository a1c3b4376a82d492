"""GPU parity of the small kernel (symmetric instances of at most 32 locations,
one warp per replica, the automatic choice there): sizes at the edges of its
compiled ranges, values of all widths, signs and diagonals, every sequential
mode, resume, more replicas than slots (parts) and the target bookkeeping.
Every replica compared equals the CPU oracle's bit for bit."""

import numpy as np
import pytest

import oracle as O
from paper_2605_24408_gb300 import instances as G

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

KEYS = ("final_perm", "final_cost", "best_perm", "best_cost", "best_sweep", "accepted")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_24408_gb300 import build as B

    B.build()
    torch.cuda.set_device(0)


def P():
    from paper_2605_24408_gb300 import pdit

    return pdit


def run(D, F, beta, S, seed, R, **kw):
    p = P()
    with p.Qap(D, F) as q:
        p.pdit_set_class_update(q, False)
        shape = p.pdit_launch_shape(q, R)
        assert shape["influence"] == "table" and shape["pending_swaps"] == 1
        out = p.anneal_device(q, R, torch.from_numpy(np.ascontiguousarray(beta, np.float32)).cuda(), S, seed,
                              per_replica=True, **kw)
        torch.cuda.synchronize()
        g = {k: v.cpu().numpy() for k, v in out.items() if k != "workspace"}
    assert int(g["status"][0]) == 0
    return g


def check(g, r, sl=slice(None)):
    for k in KEYS:
        assert np.array_equal(g["replica_" + k][sl], r[k]), k


@pytest.mark.parametrize("n", [2, 3, 12, 15, 16, 17, 24, 25, 31, 32])
def test_sizes(n):
    D, F = G.dense_instance(n, seed=n + 2)
    S = 30
    beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
    check(run(D, F, beta, S, 5, 9), O.anneal(D, F, beta, S, 5, 0, 9, threads=8))


@pytest.mark.parametrize("n,lo,hi,fmax,diag", [(12, -9, 9, 9, True), (20, 0, 3000, 900, False),
                                               (32, -127, 127, 127, True), (29, 0, 40000, 60, False)])
def test_values(n, lo, hi, fmax, diag):
    D = G.random_symmetric(n, lo, hi, seed=n, tag=3, diag=diag)
    F = G.random_symmetric(n, -fmax if lo < 0 else 0, fmax, seed=n, tag=4, diag=diag)
    S = 20
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    check(run(D, F, beta, S, 9, 6), O.anneal(D, F, beta, S, 9, 0, 6, threads=6))
    for b in (0.0, 1e30):
        beta = np.full(4, b, np.float32)
        check(run(D, F, beta, 4, 9, 3), O.anneal(D, F, beta, 4, 9, 0, 3, threads=3))


def test_modes_resume_and_target():
    D, F = G.named("n30")
    p = P()
    bm = O.beta_max(D, F)
    fb = np.array([bm * f for f in (0.0, 0.1, 1.0, 10.0)], np.float32)
    check(run(D, F, fb, 12, 2, 4, mode=p.PDIT_MODE_FIXED), O.anneal(D, F, fb, 12, 2, 0, 4, threads=4, mode="fixed"))
    ladder = O.beta_schedule("geometric", 5, bm)
    g = run(D, F, ladder, 22, 6, 10, mode=p.PDIT_MODE_PT, ladder_len=5, exchange_period=4, timeout_periods=2)
    r = O.anneal(D, F, ladder, 22, 6, 0, 10, threads=8, mode="pt", ladder_len=5, period=4, timeout=2)
    check(g, r)
    assert np.array_equal(g["replica_rung"], r["rung"])
    S, R = 60, 16
    beta = O.beta_schedule("geometric", S, bm)
    r = O.anneal(D, F, beta, S, 1, 0, R, threads=8)
    target = int(np.sort(r["best_cost"])[R // 2])
    ro = O.anneal(D, F, beta, S, 1, 0, R, threads=8, target=target)
    g = run(D, F, beta, S, 1, R, target=torch.tensor([target], dtype=torch.int64, device="cuda"))
    check(g, r)
    assert int(g["reach_sweep"][0]) == int(ro["reach_sweep"].min())
    with p.Qap(D, F) as q:
        dbeta = torch.from_numpy(beta).cuda()
        a = p.anneal_device(q, R, dbeta, S, 1, per_replica=True, sweep_end=23)
        # continued by the dot-product kernel: the state between calls is the same
        p.pdit_set_influence(q, p.PDIT_INFLUENCE_PRODUCTS)
        ws = torch.empty(1 << 22, dtype=torch.uint8, device="cuda")
        ws[:a["workspace"].numel()] = a["workspace"]
        b = p.anneal_device(q, R, dbeta, S, 1, per_replica=True, sweep_begin=23, resume=True, workspace=ws)
        torch.cuda.synchronize()
        check({k: v.cpu().numpy() for k, v in b.items() if k != "workspace"}, r)


@pytest.mark.parametrize("n", [13, 32])
def test_parts(n):
    D, F = G.dense_instance(n, seed=n + 11)
    S = 20
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    p = P()
    with p.Qap(D, F) as q:
        p.pdit_set_class_update(q, False)
        shape = p.pdit_launch_shape(q, 1 << 20)
    R = shape["ctas"] * shape["replicas_per_cta"] + 37
    g = run(D, F, beta, S, 5, R)
    for lo, hi in [(0, 3), (R - 40, R - 37), (R - 3, R)]:
        check(g, O.anneal(D, F, beta, S, 5, lo, hi, threads=3), slice(lo, hi))
