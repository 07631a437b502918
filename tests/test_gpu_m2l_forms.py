"""The two forms of the folded free-space M2L (csrc/m2l_patch.cuh): narrow
(four lanes a target, few patches) and wide (a lane a target), at orders that
leave every remainder of the chunks of source orders and, in double precision,
one and two chunks of output orders.

Double precision: against the all-pairs oracle within ten times the per-order
truncation bounds of the decay test (a tree of level 8 translates at every
level where that test's tree has three).  Single precision: within 3e-6 of the
double-precision plan of the same order and tree, as at level 4 elsewhere."""
import numpy as np
import pytest

import workloads
from tests import oracle_cache
from tests.test_gpu_fmm import P_BOUNDS, rel, run

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2507_21913_gb300 as hp  # noqa: E402


def bound(p):
    return 10 * P_BOUNDS[max(k for k in P_BOUNDS if k <= p)]


@pytest.mark.parametrize("levels", [2, 3, 5, 8])
def test_double_orders(levels):
    x, y, q, u_ref, g_ref = oracle_cache.uniform_direct(2000, 0, 1.0)
    for p in (5, 8, 11, 12, 17, 24, 25, 26, 27, 31, 40):
        u, g, _ = run(x, y, q, 1.0, p, 32, levels=levels)
        assert rel(u, u_ref) < bound(p), p
        assert rel(g, g_ref) < 30 * bound(p), p


@pytest.mark.parametrize("levels", [3, 8])
def test_single_orders(levels):
    x, y, q, _, _ = oracle_cache.uniform_direct(2000, 0, 1.0)
    for p in (12, 13, 14, 15, 16, 20, 21, 27, 40):
        u, g, _ = run(x, y, q, 1.0, p, 32, prec="fp32", levels=levels)
        u64, g64, _ = run(x, y, q, 1.0, p, 32, levels=levels)
        assert rel(u, u64) < 3e-6, p
        assert rel(g, g64) < 3e-5, p


@pytest.mark.parametrize("nrhs", [2, 33])
def test_many_vectors_take_the_wide_form(nrhs):
    """One vector at a time (narrow) and together (wide from 33 vectors on level 6)."""
    x, y, _ = workloads.uniform(20_000, seed=4)
    rng = np.random.default_rng(5)
    Q = rng.uniform(-1, 1, (nrhs, x.size))
    t = lambda a: torch.tensor(a, device="cuda:0")  # noqa: E731
    plan = hp.hpfmm_create(t(x), t(y), p=15, prec="fp32", levels=6)
    u, g = hp.hpfmm_eval(plan, t(Q))
    for r in (0, nrhs - 1):
        u1, g1 = hp.hpfmm_eval(plan, t(Q[r]))
        assert rel(u[r].cpu().numpy(), u1.cpu().numpy()) < 3e-6
        assert rel(g[r].cpu().numpy(), g1.cpu().numpy()) < 3e-5
