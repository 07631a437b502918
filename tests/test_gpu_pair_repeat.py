"""A reaction pair's value does not depend on the pairs that the lanes beside it
evaluate (csrc/special.cuh, the term count of the series): targets of one call
keep their results bit for bit when the targets between them change, their
places, and with them the order of every sum, staying the same."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2507_21913_gb300 as hp  # noqa: E402


def t(a):
    return torch.tensor(a, device="cuda:0")


@pytest.mark.parametrize("kappa", [1.0, 0.9 + 0.4j])
def test_results_do_not_depend_on_the_other_targets(kappa):
    rng = np.random.default_rng(4)
    n, m = 3, 4096
    xs, ys, q = 0.1 + 1e-3 * rng.random(n), 0.2 + 1e-3 * rng.random(n), rng.uniform(-1, 1, n)
    # |P| just below 3/4, the end of a range of one term count; |P| = 3 takes more
    r = rng.uniform(0.70, 0.745, m) / abs(kappa)
    th = rng.uniform(-0.3, 0.3, m)
    xt, yt = 0.1 + r * np.sin(th), r * np.cos(th) - 0.2
    xf, yf = xt.copy(), yt.copy()
    xf[1::2], yf[1::2] = 0.1, 2.8
    res = [hp.hpfmm_direct(t(xs), t(ys), t(q), t(a), t(b), kappa=kappa)
           for a, b in ((xt, yt), (xf, yf))]
    for a, b in zip(*res):
        assert torch.equal(torch.view_as_real(a[::2].contiguous()),
                           torch.view_as_real(b[::2].contiguous()))
