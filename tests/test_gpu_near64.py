"""The double-precision near field (csrc/near64.cu): float-pair terms up to
order 28, FP64 terms above and on one-level trees, and the lanes per target
(32 for the smallest sets down to 1).

Order 28 and order 29 differ by the far field's truncation (below 1e-12 for the
potential and 3e-11 for the gradient, the bounds that the FP64 decay test has
for order 24 with room) and by the pair arithmetic, so each configuration is
compared between the two, and with the all-pairs kernel at sampled targets."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2507_21913_gb300 as hp  # noqa: E402

POT, GRAD = 1e-12, 3e-11


def t(a):
    return torch.tensor(a, device="cuda:0")


def rel(a, b):
    return float(torch.linalg.norm(a - b) / torch.linalg.norm(b))


def evaluate(x, y, q, p, leaf, levels, kappa=1.0):
    plan = hp.hpfmm_create(t(x), t(y), kappa=kappa, p=p, leaf_size=leaf, levels=levels)
    return hp.hpfmm_eval(plan, t(q))


def points(kind, n):
    x, y, q = workloads.uniform(n, seed=n)
    if kind == "shifted":  # a small square far from the origin
        x, y = 700.0 + 1e-3 * x, 1e-3 * y
    elif kind == "close":  # pairs far closer than the fixed-point unit's reach
        m = n // 4
        x[:m] = x[m:2 * m] + 1e-13
        y[:m] = y[m:2 * m]
    elif kind == "dense":  # leaves of a thousand points beside empty ones
        x[: n // 2] = 0.4 + 0.01 * x[: n // 2]
        y[: n // 2] = 0.4 + 0.01 * y[: n // 2]
    return x, y, q


@pytest.mark.parametrize("kind,n,leaf,levels", [
    ("uniform", 3, 8, 1), ("uniform", 31, 8, 2), ("uniform", 1025, 16, 0),
    ("uniform", 4099, 32, 0), ("uniform", 20011, 16, 0), ("uniform", 65537, 32, 0),
    ("uniform", 131071, 48, 0), ("uniform", 131073, 24, 0),
    ("shifted", 3001, 24, 0), ("close", 4003, 16, 0), ("dense", 4003, 16, 4)])
def test_float_pairs_match_double_pairs(kind, n, leaf, levels):
    x, y, q = points(kind, n)
    u, g = evaluate(x, y, q, 28, leaf, levels)
    u2, g2 = evaluate(x, y, q, 29, leaf, levels)
    assert rel(u, u2) < POT and rel(g, g2) < GRAD
    if kind == "shifted":
        # the far field's box centres round to 2^-44 there, 2e-9 of a leaf side:
        # not a measure of the pairs
        return
    idx = np.linspace(0, n - 1, min(n, 64)).astype(np.int64)
    ud, gd = hp.hpfmm_direct(t(x), t(y), t(q), t(x[idx]), t(y[idx]), kappa=1.0,
                             self_index=t(idx))
    assert rel(u[idx], ud) < POT and rel(g[idx], gd) < GRAD


@pytest.mark.parametrize("k", [-300, -70, 70, 300])
def test_charge_scale_is_exact(k):
    """The split charges follow the power of two of the largest: scaling every
    charge by a power of two scales every result exactly."""
    x, y, q = workloads.uniform(3001, seed=5)
    q[::3] *= 1e-9
    u, g = evaluate(x, y, q, 16, 32, 0)
    us, gs = evaluate(x, y, np.ldexp(q, k), 16, 32, 0)
    for a, b in ((u, us), (g, gs)):
        a, b = (torch.view_as_real(v).cpu().numpy() for v in (a, b))
        assert np.array_equal(np.ldexp(a, k), b)


def test_a_plan_forgets_earlier_charges():
    """The largest charge's exponent is taken anew by every evaluation."""
    x, y, q = workloads.uniform(2503, seed=6)
    plan = hp.hpfmm_create(t(x), t(y), p=12, leaf_size=24)
    u, g = hp.hpfmm_eval(plan, t(q))
    bad = q.copy()
    bad[7] = np.inf
    ub, _ = hp.hpfmm_eval(plan, t(bad))
    assert not torch.isfinite(torch.view_as_real(ub)).all()
    hp.hpfmm_eval(plan, t(1e200 * q))
    u2, g2 = hp.hpfmm_eval(plan, t(q))
    assert torch.equal(u, u2) and torch.equal(g, g2)


@pytest.mark.parametrize("first,second", [(40, 4), (24, 12)])
def test_plans_of_several_orders(first, second):
    """A later plan of a lower order must not take shared memory from an
    earlier plan's kernels."""
    x, y, q = workloads.uniform(3001, seed=7)
    a = hp.hpfmm_create(t(x), t(y), p=first, leaf_size=32)
    u, g = hp.hpfmm_eval(a, t(q))
    b = hp.hpfmm_create(t(x), t(y), p=second, leaf_size=32)
    hp.hpfmm_eval(b, t(q))
    u2, g2 = hp.hpfmm_eval(a, t(q))
    assert torch.equal(u, u2) and torch.equal(g, g2)
