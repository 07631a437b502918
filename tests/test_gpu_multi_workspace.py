"""The workspace of many charge vectors holds what the passes read: the charges
point-major, padded to 8 or to a multiple of 16 vectors, and three arrays of
expansions."""
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2507_21913_gb300 as hp  # noqa: E402


@pytest.mark.parametrize("nrhs,padded", [(5, 8), (16, 16), (33, 48), (64, 64)])
def test_workspace(nrhs, padded):
    n, p, levels = 6000, 10, 4
    x, y, q = (torch.tensor(a, device="cuda:0") for a in workloads.uniform(n, seed=13))
    plan = hp.hpfmm_create(x, y, p=p, prec="fp32", levels=levels)
    before = plan.info()["workspace_bytes"]
    hp.hpfmm_eval(plan, q.repeat(nrhs, 1))
    boxes = (4 ** (levels + 1) - 1) // 3
    assert plan.info()["workspace_bytes"] - before == 4 * n * padded + 3 * 8 * boxes * (p + 1) * nrhs
