"""Single-precision results do not depend on the unit of length: with coordinates
scaled by a power of two and kappa by its inverse every argument kappa s keeps its
bits, and the field scales exactly (the logarithms of lengths, which do not, enter
the potential alone).  All pairs of these points have |kappa s| <= 1, where the
reaction pairs take single precision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2507_21913_gb300 as hp  # noqa: E402


def field(x, y, q, kappa, s, levels):
    t = lambda a: torch.tensor(a, device="cuda:0")  # noqa: E731
    plan = hp.hpfmm_create(t(x * s), t(y * s), kappa=kappa / s, p=12, prec="fp32", levels=levels,
                           root=(0.0, s))
    return torch.view_as_real(hp.hpfmm_eval(plan, t(q))[1]) * s


@pytest.mark.parametrize("levels", [1, 3])
@pytest.mark.parametrize("kappa", [0.4, 0.3 + 0.2j])
@pytest.mark.parametrize("k", [-40, -7, 20])
def test_field_scales(k, kappa, levels):
    rng = np.random.default_rng(5)
    x, y, q = rng.random(500), 1.0 - rng.random(500), rng.uniform(-1, 1, 500)
    assert torch.equal(field(x, y, q, kappa, 2.0 ** k, levels), field(x, y, q, kappa, 1.0, levels))


@pytest.mark.parametrize("kappa", [1e-10, 1e-16, 1e-19, 1e-25])
def test_small_kappa(kappa):
    """|P|^2 down to and below the smallest float."""
    t = lambda a: torch.tensor(a, device="cuda:0")  # noqa: E731
    rng = np.random.default_rng(6)
    x, y, q = t(rng.random(400)), t(1.0 - rng.random(400)), t(rng.uniform(-1, 1, 400))
    u, g = hp.hpfmm_eval(hp.hpfmm_create(x, y, kappa=kappa, p=16, prec="fp32", levels=2), q)
    ud, gd = hp.hpfmm_direct(x, y, q, kappa=kappa)
    for a, b, tol in ((u, ud, 5e-6), (g, gd, 5e-5)):
        assert float(torch.linalg.norm(a - b)) < tol * float(torch.linalg.norm(b))
