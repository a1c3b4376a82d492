"""GPU parity of the concurrent-update kernel (mode 3 of symmetric instances
with zero diagonals and entries in 0..127, at most 128 locations, no table
dump): sizes at the edges of its tiles, the largest entries, extreme betas,
conflicts, resume across kernels, more replicas than slots (parts) and the
target bookkeeping. Every replica compared equals the CPU oracle's bit for bit."""

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
        out = p.anneal_device(q, R, torch.from_numpy(np.ascontiguousarray(beta, np.float32)).cuda(), S, seed,
                              per_replica=True, mode=p.PDIT_MODE_CUPIM, **kw)
        torch.cuda.synchronize()
        g = {k: v.cpu().numpy() for k, v in out.items() if k != "workspace"}
    assert int(g["status"][0]) == 0
    return g


def check(g, r, sl=slice(None)):
    for k in KEYS:
        assert np.array_equal(g["replica_" + k][sl], r[k]), k


def ref(D, F, beta, S, seed, lo, hi, **kw):
    return O.anneal(D, F, beta, S, seed, lo, hi, mode="cupim", threads=8, **kw)


@pytest.mark.parametrize("n", [2, 3, 15, 16, 17, 32, 33, 48, 49, 64, 65, 80, 96, 97, 100, 112, 113, 127, 128, 129])
def test_sizes(n):
    D, F = G.dense_instance(n, seed=n + 2)
    S = 16
    beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
    check(run(D, F, beta, S, 5, 5), ref(D, F, beta, S, 5, 0, 5))


@pytest.mark.parametrize("n", [20, 128])
def test_largest_entries_and_extreme_betas(n):
    D = np.full((n, n), 127, np.int32) - G.random_symmetric(n, 0, 1, seed=n, tag=3)
    F = np.full((n, n), 127, np.int32) - G.random_symmetric(n, 0, 127, seed=n, tag=4)
    np.fill_diagonal(D, 0)
    np.fill_diagonal(F, 0)
    bm = O.beta_max(D, F)
    for beta in (np.zeros(3, np.float32), np.full(3, 1e30, np.float32), O.beta_schedule("linear", 8, bm)):
        check(run(D, F, beta, len(beta), 9, 3), ref(D, F, beta, len(beta), 9, 0, 3))


def test_hand_worked_conflicts():
    from tests import test_oracle_cupim_rule as C

    beta = np.array([C.BIG_BETA], np.float32)
    g = run(C.D, C.F, beta, 1, C.SEED, 1)
    check(g, ref(C.D, C.F, beta, 1, C.SEED, 0, 1))
    assert g["replica_final_perm"][0].tolist() == C.EXPECTED


def test_resume_and_target():
    D, F = G.dense_instance(75, seed=4)
    S, R = 40, 8
    p = P()
    beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
    r = ref(D, F, beta, S, 1, 0, R)
    target = int(np.sort(r["best_cost"])[R // 2])
    ro = ref(D, F, beta, S, 1, 0, R, target=target)
    g = run(D, F, beta, S, 1, R, target=torch.tensor([target], dtype=torch.int64, device="cuda"))
    check(g, r)
    assert int(g["reach_sweep"][0]) == int(ro["reach_sweep"].min())
    with p.Qap(D, F) as q:
        dbeta = torch.from_numpy(beta).cuda()
        ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
        kw = dict(per_replica=True, mode=p.PDIT_MODE_CUPIM, workspace=ws)
        p.anneal_device(q, R, dbeta, S, 1, sweep_end=13, **kw)
        p.pdit_set_influence(q, p.PDIT_INFLUENCE_TABLE)  # the table kernels carry on
        p.anneal_device(q, R, dbeta, S, 1, sweep_begin=13, sweep_end=21, resume=True, **kw)
        p.pdit_set_influence(q, p.PDIT_INFLUENCE_AUTO)
        b = p.anneal_device(q, R, dbeta, S, 1, sweep_begin=21, resume=True, **kw)
        torch.cuda.synchronize()
        check({k: v.cpu().numpy() for k, v in b.items() if k != "workspace"}, r)


@pytest.mark.parametrize("n,R", [(12, 6000), (100, 701)])
def test_parts(n, R):
    D, F = G.dense_instance(n, seed=n + 11)
    S = 20
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    g = run(D, F, beta, S, 5, R)
    for lo, hi in [(0, 3), (R // 2, R // 2 + 3), (R - 3, R)]:
        check(g, ref(D, F, beta, S, 5, lo, hi), slice(lo, hi))
