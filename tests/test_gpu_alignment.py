"""Complex arrays of the C ABI aligned to a double and no more, as C's double
_Complex is: the results of aligned arrays, or EINVAL from single-precision plans
on the uniform tree.  (PyTorch's complex tensors are aligned to 16 bytes.)"""
import ctypes

import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2507_21913_gb300 as hp  # noqa: E402

N = 3001


def t(a):
    return torch.tensor(a, device="cuda:0")


class Odd:
    """m doubles at an address 8 beyond a multiple of 16, and the doubles around."""

    def __init__(self, m):
        self.all = torch.full((m + 4,), 7.25, dtype=torch.float64, device="cuda:0")
        self.v = self.all[1:m + 1]
        self.ptr = self.all.data_ptr() + 8
        assert self.ptr % 16 == 8

    def whole(self):
        return self.v.clone()

    def untouched(self):
        return bool((self.all[:1] == 7.25).all() and (self.all[1 + len(self.v):] == 7.25).all())


def real(a):
    return torch.view_as_real(a.contiguous()).reshape(-1)


def call(name, *args):
    args = [ctypes.c_void_p(a) if isinstance(a, int) and a > 1 << 20 else a for a in args]
    hp._check(getattr(hp.lib(), name)(*args, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))


def check(pairs):
    torch.cuda.synchronize()
    for odd, ref in pairs:
        assert torch.equal(odd.whole(), ref) and odd.untouched()


@pytest.mark.parametrize("prec,adaptive,nrhs", [("fp64", False, 1), ("mixed", True, 1),
                                                ("fp64", False, 2)])
@pytest.mark.parametrize("grad", [True, False])
def test_eval(prec, adaptive, nrhs, grad):
    x, y, q = workloads.uniform(N, seed=8)
    q = t(q).repeat(nrhs, 1) * torch.arange(1, nrhs + 1, device="cuda:0")[:, None]
    plan = hp.hpfmm_create(t(x), t(y), p=12, prec=prec, adaptive=adaptive)
    u, g = hp.hpfmm_eval(plan, q, grad=grad)
    po, go = Odd(2 * nrhs * N), Odd(4 * nrhs * N)
    call("hpfmm_eval", plan.handle, q.data_ptr(), nrhs, po.ptr, go.ptr if grad else None)
    check([(po, real(u))] + ([(go, real(g))] if grad else []))


@pytest.mark.parametrize("nrhs", [1, 3])
def test_uniform_single_precision_refuses(nrhs):
    x, y, q = (t(a) for a in workloads.uniform(N, seed=8))
    q = q.repeat(nrhs, 1)
    plan = hp.hpfmm_create(x, y, p=12, prec="fp32")
    po, go = Odd(2 * nrhs * N), Odd(4 * nrhs * N)
    u, g = hp.hpfmm_eval(plan, q)
    for pot, grad in ((po.ptr, None), (po.ptr, go.ptr), (u.data_ptr(), go.ptr)):
        with pytest.raises(hp.HpfmmError) as e:
            call("hpfmm_eval", plan.handle, q.data_ptr(), nrhs, pot, grad)
        assert e.value.status == hp.HPFMM_EINVAL
    b = hp.hpfmm_batch_create([plan])
    one = lambda p: (ctypes.c_void_p * 1)(p)  # noqa: E731
    with pytest.raises(hp.HpfmmError) as e:
        call("hpfmm_eval_batched", b.handle, one(q.data_ptr()), one(po.ptr), None)
    assert e.value.status == hp.HPFMM_EINVAL
    u2, g2 = hp.hpfmm_eval(plan, q)
    check([])
    assert po.untouched() and go.untouched() and torch.equal(u, u2) and torch.equal(g, g2)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_targets(prec):
    x, y, q = workloads.uniform(N, seed=9)
    xt, yt, _ = workloads.uniform(777, seed=10)
    x, y, q, xt, yt = t(x), t(y), t(q), t(xt) * 0.9 + 0.05, t(yt) * 0.9
    plan = hp.hpfmm_create(x, y, p=12, prec=prec, root=(-0.1, 1.2))
    u, g = hp.hpfmm_eval_targets(plan, q, xt, yt)
    po, go = Odd(2 * 777), Odd(4 * 777)
    call("hpfmm_eval_targets", plan.handle, q.data_ptr(), xt.data_ptr(), yt.data_ptr(), 777, po.ptr,
         go.ptr)
    check([(po, real(u)), (go, real(g))])


def test_adjoint_and_direct():
    x, y, q = (t(a) for a in workloads.uniform(N, seed=11))
    plan = hp.hpfmm_create(x, y, p=12, prec="fp32")
    _, gq = hp.hpfmm_eval(plan, q)
    c = torch.complex(torch.sin(q), torch.cos(3 * q))
    dq, dxy = hp.hpfmm_eval_adjoint(plan, q, c, grad_q=gq)
    co, gqo, dxyo = Odd(2 * N), Odd(4 * N), Odd(2 * N)
    co.v.copy_(real(c))
    gqo.v.copy_(real(gq))
    dq2 = torch.empty_like(dq)
    call("hpfmm_eval_adjoint", plan.handle, q.data_ptr(), co.ptr, gqo.ptr, dq2.data_ptr(), dxyo.ptr)
    check([(dxyo, dxy.reshape(-1))])
    assert torch.equal(dq, dq2)
    xt, yt = x[:50] * 0.9 + 0.01, y[:50] * 0.9
    u, g = hp.hpfmm_direct(x, y, q, xt, yt)
    po, go = Odd(100), Odd(200)
    call("hpfmm_direct", x.data_ptr(), y.data_ptr(), q.data_ptr(), N, xt.data_ptr(), yt.data_ptr(),
         None, 50, 1.0, 0.0, po.ptr, go.ptr)
    check([(po, real(u)), (go, real(g))])


def test_batch():
    plans, qs = [], []
    for k, n in enumerate((500, 1201)):
        x, y, q = (t(a) for a in workloads.uniform(n, seed=k))
        plans.append(hp.hpfmm_create(x, y, p=10, prec="fp64"))
        qs.append(q)
    b = hp.hpfmm_batch_create(plans)
    us, gs = hp.hpfmm_eval_batched(b, qs)
    us, gs = [u.clone() for u in us], [g.clone() for g in gs]
    po, go = [Odd(2 * p.n) for p in plans], [Odd(4 * p.n) for p in plans]
    arr = lambda ptrs: (ctypes.c_void_p * 2)(*ptrs)  # noqa: E731
    call("hpfmm_eval_batched", b.handle, arr([q.data_ptr() for q in qs]), arr([o.ptr for o in po]),
         arr([o.ptr for o in go]))
    check([(o, real(u)) for o, u in zip(po, us)] + [(o, real(g)) for o, g in zip(go, gs)])
