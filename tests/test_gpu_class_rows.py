"""The flow-class kernel's row loads: rows of D of 1, 2 and 4 bytes an entry,
one to eight candidates a thread, at sizes whose rows end inside a word."""

import pytest

import oracle as O
from gpu_common import check, device, host, library
from paper_2605_24408_gb300 import instances as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top", [99, 3000, 40000])
@pytest.mark.parametrize("n,wpr", [(33, 1), (61, 1), (61, 2), (121, 1), (127, 2), (128, 4), (201, 1), (229, 2),
                                   (230, 4), (231, 8)])
def test_rows(n, wpr, top):
    p = library()
    D, F = G.flow_class_instance(n, n // 3, seed=n + wpr, hi=top)
    S, R = 5, 6
    beta = O.beta_schedule("geometric", S, O.beta_max(D, F))
    with p.Qap(D, F) as q:
        assert p.pdit_instance_form(q) == p.PDIT_FORM_FLOW_CLASSES
        p.pdit_set_warps_per_replica(q, wpr)
        g = host(p.anneal_device(q, R, device(beta), S, 8, per_replica=True))
    check(g, O.anneal(D, F, beta, S, 8, 0, R, threads=6))
