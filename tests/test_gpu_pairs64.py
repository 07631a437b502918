"""Pairs of the double-precision near field (csrc/near64.cu) point by point:
integer pairs (order 28) against FP64 pairs (order 29).

All points lie in neighbouring leaves and closer to one another than a
thousandth of a leaf side, so that the near field is 1e3 and more times the far
field, whose truncation (below 1e-12 of it) then stays below 1e-15 of the sums of
the terms' magnitudes that the bounds count in.  FP64 terms round four times and
their sum of n once each: (4 + n) 2^-53; the integer pairs add 2^-53, the scaling
of the result another."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2507_21913_gb300 as hp  # noqa: E402

LEVELS, ROOT = 3, (-0.5, 1.0)  # leaves of 1/8


def t(a):
    return torch.tensor(a, device="cuda:0")


def points(kind, n, rng):
    """x, y in two leaves beside x = 0, most doubles finer than 2^-60 of a leaf side."""
    tiny = 2.0 ** -rng.uniform(10, 60, n)
    u, v = rng.uniform(-1e-4, 1e-4, n), np.sort(rng.uniform(0, 1e-4, n))
    if kind == "column at x = 0":
        return tiny * 1e-5 * rng.choice([-1, 1], n), 0.3 + v
    if kind == "next to y = 0":
        return 0.05 + u, tiny * 1e-2
    if kind == "corner":
        return u * tiny * 1e3, v * tiny * 1e3 + 1e-20
    return 0.05 + u, 0.3 + v


def evaluate(x, y, q, p):
    plan = hp.hpfmm_create(t(x), t(y), p=p, leaf_size=8, levels=LEVELS, root=ROOT)
    u, g = hp.hpfmm_eval(plan, t(q))
    return u.cpu().numpy(), g.cpu().numpy()


def magnitudes(x, y, q):
    r = np.hypot(x[:, None] - x[None], y[:, None] - y[None])
    np.fill_diagonal(r, 1.0)
    w = np.abs(q)[None] * (1 - np.eye(len(x))) / (2 * np.pi)
    return (w * np.maximum(1, np.abs(np.log(r)))).sum(1), (w / r).sum(1)


@pytest.mark.parametrize("n", [2, 33, 300])
@pytest.mark.parametrize("kind", ["ordinary", "column at x = 0", "next to y = 0", "corner"])
def test_points_match_double_pairs(kind, n):
    rng = np.random.default_rng(n)
    x, y = points(kind, n, rng)
    q = rng.uniform(-1, 1, n)
    q[::5] *= 2.0 ** -20
    (u, g), (u2, g2) = evaluate(x, y, q, 28), evaluate(x, y, q, 29)
    mu, mg = magnitudes(x, y, q)
    tol = (n + 6) * 2.0 ** -53
    # the image and reaction sums (the same in both) round the gradient's total too
    assert (np.abs(u - u2) <= tol * mu + 1e-12 * np.abs(q).sum()).all()
    assert (np.abs(g - g2).max(1) <= tol * (mg + np.abs(g2).max(1)) + 1e-11 * np.abs(q).sum()).all()


@pytest.mark.parametrize("scale", [2.0 ** -1040, 2.0 ** -1022, 2.0 ** 900])
def test_charges_at_the_ends_of_the_range(scale):
    """Subnormal charges give FP64 pairs, which keep what their bits hold."""
    rng = np.random.default_rng(3)
    x, y = points("ordinary", 60, rng)
    q = rng.uniform(-1, 1, 60) * scale
    (u, g), (u2, g2) = evaluate(x, y, q, 28), evaluate(x, y, q, 29)
    mu, mg = magnitudes(x, y, q)
    small = 60 * 2.0 ** -1074 * 16 * 1e4  # a subnormal's unit, by the largest 1 / r^2 r
    assert (np.abs(u - u2) <= 66 * 2.0 ** -53 * mu + 1e-12 * np.abs(q).sum() + small).all()
    assert (np.abs(g - g2).max(1) <= 66 * 2.0 ** -53 * (mg + np.abs(g2).max(1)) +
            1e-11 * np.abs(q).sum() + small * 1e4).all()
    assert np.abs(g2).max() > 10 * scale
