"""What the GPU tests of one kernel or one rule share: the library, a call
with per-replica outputs, and the comparison with the CPU oracle."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

KEYS = ("final_perm", "final_cost", "best_perm", "best_cost", "best_sweep", "accepted")


def library():
    """The binding, with the library built for this machine."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_24408_gb300 import build, pdit

    build.build()
    torch.cuda.set_device(0)
    return pdit


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def device(beta):
    return torch.from_numpy(np.ascontiguousarray(beta, np.float32)).cuda()


def host(out):
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items() if k != "workspace"}


def check(g, r, sl=slice(None)):
    """Replicas `sl` of a call equal the oracle's, and every audit passed."""
    assert int(g["status"][0]) == 0
    for k in KEYS:
        assert np.array_equal(g["replica_" + k][sl], r[k]), k
