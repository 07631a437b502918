"""Single-precision near field of uniform trees with leaves that overflow the
staging buffer of 1280 points (csrc/fmm.cu, k_near32): patches just below and
above one, two and three buffers, from 4 x 4 tiles (levels 4) and 2 x 2 tiles
(levels 3), with coincident points, against the all-pairs kernel to the bounds of
the other single-precision tests, and at no more cost than the pairs account for."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2507_21913_gb300 as hp  # noqa: E402


def t(a):
    return torch.tensor(a, device="cuda:0")


def rel(a, b):
    return float(torch.linalg.norm(a - b) / torch.linalg.norm(b))


def problem(dense, levels, rest=600, seed=1):
    """`rest` points everywhere and `dense` in one leaf and its right neighbour."""
    rng = np.random.default_rng(seed)
    n, d = rest + dense, 2.0 ** -levels
    x, y = rng.random(n), 1.0 - rng.random(n)
    ix = 2 ** levels // 2 - 1  # its neighbour lies in another tile
    x[:dense] = (ix + 2 * rng.random(dense) ** 3) * d
    y[:dense] = (ix + rng.random(dense)) * d
    return x, y, rng.uniform(-1, 1, n)


def plan_of(x, y, levels):
    return hp.hpfmm_create(t(x), t(y), kappa=1.0, p=16, prec="fp32", levels=levels,
                           root=(0.0, 1.0))


@pytest.mark.parametrize("levels", [3, 4])
@pytest.mark.parametrize("dense", [1200, 1279, 1281, 1800, 2559, 2562, 3900])
def test_against_all_pairs(dense, levels):
    x, y, q = problem(dense, levels)
    x[10:20], y[10:20] = x[30:40], y[30:40]  # coincident points contribute nothing
    q[10:20] = 0.0
    plan = plan_of(x, y, levels)
    u, g = hp.hpfmm_eval(plan, t(q))
    keep = np.setdiff1d(np.arange(len(x)), np.r_[10:20, 30:40])
    idx = keep[:: max(1, len(keep) // 300)]
    src = np.setdiff1d(np.arange(len(x)), np.r_[10:20])
    at = np.searchsorted(src, idx)
    ud, gd = hp.hpfmm_direct(t(x[src]), t(y[src]), t(q[src]), t(x[idx]), t(y[idx]), kappa=1.0,
                             self_index=t(at))
    assert rel(u[idx], ud) < 5e-6 and rel(g[idx], gd) < 5e-5


def test_cost_follows_the_pairs():
    """1800 points in a leaf are 3.2 times the pairs of 1000; read from global
    memory they took 29 times as long."""
    ms = {}
    for dense in (1000, 1800):
        x, y, q = problem(dense, 4, rest=4000 - dense)
        plan, qd = plan_of(x, y, 4), t(q)
        best = 1e9
        for _ in range(12):
            torch.cuda.synchronize()
            a = time.perf_counter()
            hp.hpfmm_eval(plan, qd)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - a)
        ms[dense] = best
    assert ms[1800] < 8 * ms[1000]
