"""GPU parity of the tensor-core product kernel (instances with zero diagonals
and entries in 0..127, symmetric or general, above the sizes of the small kernel):
sizes at the edges of its compiled ranges, blocks with one replica, with a
part of their slots and with all of them, entries at the ends of their range,
and where the automatic choice takes it. Every replica compared equals the
CPU oracle's bit for bit."""

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


def run(D, F, beta, S, seed, R):
    p = P()
    with p.Qap(D, F) as q:
        p.pdit_set_class_update(q, False)
        shape = p.pdit_launch_shape(q, R)
        assert shape["influence"] == "products"
        out = p.anneal_device(q, R, torch.from_numpy(beta).cuda(), S, seed, per_replica=True)
        torch.cuda.synchronize()
        g = {k: v.cpu().numpy() for k, v in out.items() if k != "workspace"}
    assert int(g["status"][0]) == 0
    return g, shape


def check(g, D, F, beta, S, seed, lo, hi):
    r = O.anneal(D, F, beta, S, seed, lo, hi, threads=min(8, hi - lo))
    for k in KEYS:
        assert np.array_equal(g["replica_" + k][lo:hi], r[k]), k


@pytest.mark.parametrize("n", [33, 48, 49, 64, 65, 80, 81, 96, 97, 112, 113, 128, 129, 160, 161, 192, 193, 224, 225, 256])
def test_size_edges(n):
    D, F = G.dense_instance(n, seed=n)
    S = 4
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    g, _ = run(D, F, beta, S, 3, 5)
    check(g, D, F, beta, S, 3, 0, 5)


@pytest.mark.parametrize("n,per_sm", [(40, 1), (75, 2), (100, 8), (100, 9), (100, 16), (100, 27), (128, 17), (150, 3),
                                      (256, 9), (256, 14)])
def test_block_fill(n, per_sm):
    """Blocks with some or all slots in use: replicas of the first block, of a
    middle one and of the last (short) one."""
    D, F = G.dense_instance(n, seed=n + 1)
    S = 3
    beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    R = sms * per_sm - per_sm // 2
    g, _ = run(D, F, beta, S, 8, R)
    for lo, hi in ((0, min(R, 32)), (R // 2, R // 2 + 4), (R - 6, R)):
        check(g, D, F, beta, S, 8, lo, hi)


@pytest.mark.parametrize("hi", [1, 127])
def test_entry_range(hi):
    """Entries all at the top of the range (the largest products and sums) or
    0 and 1 (many equal energies), and the beta extremes."""
    n, S = 113, 6
    D = G.random_symmetric(n, hi if hi > 1 else 0, hi, seed=1, tag=3)
    F = G.random_symmetric(n, 0, hi, seed=2, tag=5)
    for beta in (O.beta_schedule("linear", S, O.beta_max(D, F)), np.zeros(S, np.float32),
                 np.full(S, 1e30, np.float32)):
        g, _ = run(D, F, beta, S, 4, 6)
        check(g, D, F, beta, S, 4, 0, 6)


@pytest.mark.parametrize("n", [33, 48, 49, 64, 65, 80, 81, 96, 97, 112, 113, 128, 129, 160])
def test_general_form_size_edges(n):
    D, F = G.asymmetric(n, 0, 99, n, 101), G.asymmetric(n, 0, 99, n, 103)
    S = 5
    beta = O.beta_schedule("linear", S, O.beta_max(D, F))
    g, _ = run(D, F, beta, S, 3, 5)
    check(g, D, F, beta, S, 3, 0, 5)


@pytest.mark.parametrize("n,per_sm", [(50, 9), (100, 27), (120, 3), (150, 12)])
def test_general_form_block_fill(n, per_sm):
    D, F = G.asymmetric_instance(n, seed=n)
    S = 3
    beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    R = sms * per_sm - per_sm // 2
    g, _ = run(D, F, beta, S, 8, R)
    for lo, hi in ((0, min(R, 32)), (R // 2, R // 2 + 4), (R - 6, R)):
        check(g, D, F, beta, S, 8, lo, hi)
