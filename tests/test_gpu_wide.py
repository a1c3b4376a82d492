"""GPU parity of the product kernel's wide form (symmetric instances with zero
diagonals and entries in 0..2047, some above 127; 33 to 128 locations): sizes
at the edges of its compiled ranges, the largest entries, extreme betas, block
fills, parts, the other sequential modes, resume across kernels and a batch.
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


def wide(n, top, seed, low=0):
    return G.dense_symmetric(n, low, top, seed, tag=23), G.dense_symmetric(n, low, top, seed, tag=33)


def host(out):
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items() if k != "workspace"}


def run(D, F, beta, S, seed, R, products=True, **kw):
    p = P()
    with p.Qap(D, F) as q:
        # (a call of the product kernel keeps no tables between its segments)
        o = p.opts(replicas=R, sweeps=S, mode=p.PDIT_MODE_PT, ladder_len=R) if 2 <= R <= 64 else None
        if o is not None:
            need = p.pdit_workspace_bytes(q, o)
            assert (need < R * len(D) * len(D) * 4) == products
        g = host(p.anneal_device(q, R, torch.from_numpy(np.ascontiguousarray(beta, np.float32)).cuda(), S, seed,
                                 per_replica=True, **kw))
    assert int(g["status"][0]) == 0
    return g


def check(g, r, sl=slice(None)):
    for k in KEYS:
        assert np.array_equal(g["replica_" + k][sl], r[k]), k


@pytest.mark.parametrize("n", [33, 48, 49, 61, 64, 65, 80, 81, 96, 97, 112, 113, 120, 128])
def test_size_edges(n):
    D, F = wide(n, 999, n)
    S = 6
    beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
    check(run(D, F, beta, S, 3, 5), O.anneal(D, F, beta, S, 3, 0, 5, threads=5))


@pytest.mark.parametrize("n,top,low,ftop,products", [(33, 2047, 2000, 1800, True), (33, 1800, 1790, 2047, True),
                                                     (33, 2048, 0, 1800, False), (128, 1010, 1000, 1010, True),
                                                     (50, 128, 0, 1, True)])
def test_entry_range_and_extreme_betas(n, top, low, ftop, products):
    D, _ = wide(n, top, 7, low)
    _, F = wide(n, ftop, 7, min(low, ftop - 10) if ftop > 10 else 0)
    D[0, 1] = D[1, 0] = top
    for beta in (O.beta_schedule("linear", 6, O.beta_max(D, F)), np.zeros(4, np.float32), np.full(4, 1e30, np.float32)):
        S = len(beta)
        check(run(D, F, beta, S, 4, 5, products), O.anneal(D, F, beta, S, 4, 0, 5, threads=5))


@pytest.mark.parametrize("n,per_sm", [(40, 1), (61, 4), (75, 9), (100, 16), (100, 27), (128, 17), (61, 60)])
def test_block_fill_and_parts(n, per_sm):
    D, F = wide(n, 999, n + 1)
    S = 9
    beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
    R = torch.cuda.get_device_properties(0).multi_processor_count * per_sm - per_sm // 2
    g = run(D, F, beta, S, 8, R)
    for lo, hi in ((0, 8), (R // 2, R // 2 + 4), (R - 6, R)):
        check(g, O.anneal(D, F, beta, S, 8, lo, hi, threads=8), slice(lo, hi))


def test_modes_resume_and_batch():
    D, F = wide(61, 999, 2)
    p = P()
    bm = O.beta_max(D, F)
    fb = np.array([bm * f for f in (0.0, 0.1, 1.0, 10.0)], np.float32)
    check(run(D, F, fb, 8, 2, 4, mode=p.PDIT_MODE_FIXED), O.anneal(D, F, fb, 8, 2, 0, 4, threads=4, mode="fixed"))
    ladder = O.beta_schedule("geometric", 5, bm)
    g = run(D, F, ladder, 14, 6, 10, mode=p.PDIT_MODE_PT, ladder_len=5, exchange_period=4, timeout_periods=2)
    check(g, O.anneal(D, F, ladder, 14, 6, 0, 10, threads=8, mode="pt", ladder_len=5, period=4, timeout=2))
    S, R = 24, 6
    beta = O.beta_schedule("linear", S, bm)
    r = O.anneal(D, F, beta, S, 1, 0, R, threads=6)
    with p.Qap(D, F) as q:
        dbeta = torch.from_numpy(beta).cuda()
        ws = torch.empty(1 << 22, dtype=torch.uint8, device="cuda")
        kw = dict(per_replica=True, workspace=ws)
        p.anneal_device(q, R, dbeta, S, 1, sweep_end=7, **kw)
        p.pdit_set_influence(q, p.PDIT_INFLUENCE_TABLE)
        p.anneal_device(q, R, dbeta, S, 1, sweep_begin=7, sweep_end=15, resume=True, **kw)
        p.pdit_set_influence(q, p.PDIT_INFLUENCE_AUTO)
        check(host(p.anneal_device(q, R, dbeta, S, 1, sweep_begin=15, resume=True, **kw)), r)
    insts = [wide(n, 999, n) if k % 2 else G.dense_instance(n, n) for k, n in enumerate((61, 61, 64, 100, 40))]
    items, want = [], []
    for k, (A, B) in enumerate(insts):
        b = O.beta_schedule("linear", S, O.beta_max(A, B))
        items.append({"qap": p.Qap(A, B), "replicas": 20, "sweeps": S, "beta": torch.from_numpy(b).cuda(), "seed": 3,
                      "instance_id": k})
        want.append(O.anneal(A, B, b, S, 3, 0, 20, threads=8, inst=k))
    batch = p.Batch(items)
    batch.run()
    torch.cuda.synchronize()
    for o, r in zip(batch.out, want):
        assert int(o["best_cost"].item()) == r["cost"]
        assert np.array_equal(o["best_perm"].cpu().numpy(), r["perm"])
