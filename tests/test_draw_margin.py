"""The binary32 draw that stands in front of the exact one (eq5_draw_core in
pdit_sweep.cuh) keeps an outcome only if the draw lies further than 2^-16 of
the total from its interval's ends. On the CPU: a binary32 model of that draw,
with ex2.approx off by its full documented error in the worst directions,
against the oracle's integer weights. Its prefix shares stay within the
margin, and every outcome it keeps is the exact one, with draws placed
at the interval ends as well as at random."""

import numpy as np
import pytest

import oracle as O

F32 = np.float32
MARGIN = 2.0 ** -16


def exact_prefix(dE, beta):
    d = dE - dE.min()
    x = d.astype(F32) * F32(beta)
    w = [O.weight(float(v)) for v in x]
    return np.cumsum(np.array(w, dtype=object))


def model_prefix(dE, beta, err):
    """Thread-contiguous binary32 sums as the kernels form them: per thread,
    then a 32-lane scan (one warp holds up to 8 outcomes a lane)."""
    n = len(dE)
    k = max(1, 1 << int(np.ceil(np.log2(max(n, 32) / 32))))
    kb = F32(-F32(beta) * F32(1.44269502))
    arg = dE.astype(F32) * kb
    w = (np.exp2(arg.astype(np.float64)) * (1.0 + err * 2.0 ** -22)).astype(F32)
    full = np.zeros(32 * k, F32)
    full[:n] = w
    pre = np.cumsum(full.reshape(32, k), axis=1, dtype=F32)
    incl = pre[:, -1].copy()
    for o in (1, 2, 4, 8, 16):
        y = np.concatenate([np.zeros(o, F32), incl[:-o]])
        incl = incl + y
    excl = incl - pre[:, -1]
    return (excl[:, None] + pre).reshape(-1)[:n], incl[-1]


@pytest.mark.parametrize("n", [2, 12, 33, 100, 256])
@pytest.mark.parametrize("top", [0.0, 0.5, 5.0, 44.0])  # beta x the largest downhill energy
def test_kept_outcomes_are_exact(n, top):
    rng = np.random.default_rng(n * 100 + int(top))
    for trial in range(8):
        scale = int(10 ** rng.uniform(1, 6.3))
        dE = rng.integers(-scale if top else 0, 4 * scale, n).astype(np.int64)
        dE[rng.integers(n)] = 0  # the stay outcome
        low = max(1, -int(dE.min()))
        beta = F32(top / low if top else rng.choice([0.0, 1e-7, 1.0 / scale, 20.0 / scale]))
        P = exact_prefix(dE, beta)
        T = int(P[-1])
        share = np.array([float(p) / float(T) for p in P])
        for err in (rng.uniform(-1, 1, n), np.sign(np.arange(n) - rng.integers(n))):
            pre, total = model_prefix(dE, beta, err)
            if not total < 2.0 ** 64:
                continue  # the kernels keep nothing then
            off = np.abs(pre.astype(np.float64) / float(total) - share).max()
            assert off < MARGIN, off
            # draws at the ends of intervals (where a wrong pick would
            # happen) and at random
            draws = [int(rng.integers(0, 2 ** 64, dtype=np.uint64)) for _ in range(20)]
            for p in P[rng.integers(0, n, 20)]:
                for eps in (-3e-5, -1e-6, 0.0, 1e-6, 3e-5):
                    draws.append(min(2 ** 64 - 1, max(0, int((float(p) / T + eps) * 2.0 ** 64))))
            m = F32(MARGIN) * total
            lo = np.concatenate([[F32(0)], pre[:-1]])
            for r in draws:
                tt = F32(F32((r >> 40)) * F32(2.0 ** -24)) * total
                kept = np.flatnonzero((tt - m >= lo) & (tt + m < pre))
                exact = int(np.searchsorted(P, (r * T) >> 64, side="right"))
                assert len(kept) <= 1
                if len(kept):
                    assert int(kept[0]) == exact
