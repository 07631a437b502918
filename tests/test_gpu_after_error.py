"""A double-precision plan after an evaluation that failed between its gather and
its downward pass: the next one does not take that one's largest charge.

The failure is an error code on the host: hpfmm_sync waits for a stream under
capture, which the runtime refuses, and the next call's launch check reports the
pending code after its first kernels."""
import ctypes

import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2507_21913_gb300 as hp  # noqa: E402


def refused_wait(plan):
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        g.capture_begin(capture_error_mode="thread_local")
        status = hp.lib().hpfmm_sync(plan.handle, ctypes.c_void_p(s.cuda_stream))
        try:
            g.capture_end()
        except RuntimeError:
            pass
    assert status == hp.HPFMM_ECUDA


def test_the_largest_charge_of_a_failed_evaluation_is_forgotten():
    t = lambda a: torch.tensor(a, device="cuda:0")  # noqa: E731
    x, y, q = (t(a) for a in workloads.uniform(3001, seed=12))
    plan = hp.hpfmm_create(x, y, p=12, leaf_size=24)
    hp.hpfmm_sync(plan)
    u, g = hp.hpfmm_eval(plan, q)
    torch.cuda.synchronize()
    refused_wait(plan)
    with pytest.raises(hp.HpfmmError) as e:
        hp.hpfmm_eval(plan, 1e200 * q)
    assert e.value.status == hp.HPFMM_ECUDA
    u2, g2 = hp.hpfmm_eval(plan, q)
    assert torch.equal(u, u2) and torch.equal(g, g2)
