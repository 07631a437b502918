"""The work that users of the half-plane Robin FMM have it do, as measured cases.

A case is one call pattern of the public entry points at one size:

* ``eval``     potentials (and fields) on a kept plan: the matrix-vector product
               of an iterative solver, or repeated charges on fixed points
* ``step``     moving points: the plan's tree and tables rebuilt in place, then
               potentials and fields
* ``adjoint``  one differentiable call and its backward pass (charges and positions)
* ``rhs``      many charge vectors on one point set
* ``batch``    independent problems of uneven size as one call
* ``targets``  field points that are not sources (charged circles and a mesh)
* ``direct``   the all-pairs sum at sampled targets, the check of an FMM result

``listed()`` names the sizes in use; ``draw()`` covers the ranges around them.

Single-precision plans ("fp32", "mixed") hand their results back in
double-precision storage that holds single-precision numbers.  A program that
asks for single precision goes on in it, so ``run`` converts such results to
complex64 / float32.  Double-precision results are returned as they are.

``exact`` sums the kernel directly in double precision, with the exponential
integral's power series, wherever that takes some seconds.
"""
import math

import numpy as np
import torch

import paper_2507_21913_gb300 as hp

TWO_PI = 2.0 * math.pi
EULER_GAMMA = 0.57721566490153286061

# pairs x series terms of a direct double-precision sum that exact() may spend
EXACT_BUDGET = 4e11


def listed():
    return [
        # the smallest solver call: the paper-sized problem of 2000 points in
        # double precision, where launches and latency are all there is
        dict(name="solve_2k_fp64", kind="eval", shape="uniform", n=2000, kre=1.0, kim=0.0, p=12,
             leaf=32, prec="fp64", grad=True),
        # a small ragged cloud that moves every step
        dict(name="move_7k_fp32", kind="step", shape="uniform", n=7321, kre=0.7, kim=0.0, p=13,
             leaf=32, prec="fp32", grad=True, wait=True),
        # high-accuracy solve at a lossy boundary, double precision, high order
        dict(name="solve_40k_fp64_p24", kind="eval", shape="uniform", n=40009, kre=1.0, kim=0.5,
             p=24, leaf=32, prec="fp64", grad=True),
        # potentials only, as a Krylov solver asks for them, at a large Robin parameter
        dict(name="matvec_50k_fp32_pot", kind="eval", shape="uniform", n=50021, kre=10.0, kim=0.0,
             p=16, leaf=32, prec="fp32", grad=False),
        # the headline step: a million moving points, single precision
        dict(name="step_1m_fp32", kind="step", shape="uniform", n=1_000_000, kre=1.0, kim=0.0,
             p=13, leaf=16, prec="fp32", grad=True, wait=False),
        # the plain double-precision FMM on the same points
        dict(name="step_1m_fp64", kind="step", shape="uniform", n=1_000_000, kre=1.0, kim=0.0,
             p=12, leaf=16, prec="fp64", grad=True, wait=True),
        # clustered points near the boundary on the adaptive tree, lossy kappa,
        # mixed precision: the largest point set
        dict(name="clustered_4m_mixed", kind="step", shape="clustered", n=4_000_000, kre=1.0,
             kim=0.5, p=20, leaf=32, prec="mixed", grad=True, wait=True),
        # a training step: forward and backward through the autograd function
        dict(name="adjoint_1m_fp32", kind="adjoint", shape="uniform", n=1_000_000, kre=2.0,
             kim=0.0, p=16, leaf=64, prec="fp32"),
        # many charge vectors on one point set
        dict(name="rhs64_500k_fp32", kind="rhs", shape="uniform", n=500_000, kre=1.0, kim=0.0,
             p=16, leaf=32, prec="fp32", nrhs=64, mode=0),
        # independent problems of uneven size, one call
        dict(name="batch32_fp32", kind="batch", count=32, lo=10_000, hi=400_000, p=16, leaf=32,
             prec="fp32"),
        # the paper's charged circles seen from a mesh of field points
        dict(name="targets_200k_125k", kind="targets", per_circle=25_000, nfx=500, nfy=250,
             kre=1.0, kim=0.0, p=16, leaf=3, prec="fp32"),
        # sampled error check of a large result: 256 targets against every source
        dict(name="check_256_of_200k", kind="direct", nt=256, n=200_003, kre=1.0, kim=0.0),
    ]


def _logint(rng, lo, hi):
    """An integer between lo and hi, spread over the logarithm, odd sizes among them."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _kappa(rng, top=10.0):
    """Robin parameters from 0.1 to `top`; one in three lossy."""
    kre = round(math.exp(rng.uniform(math.log(0.1), math.log(top))), 4)
    kim = round(rng.uniform(0.1, 0.5) * kre, 4) if rng.random() < 1 / 3 else 0.0
    return dict(kre=kre, kim=kim)


def draw(rng):
    kind = rng.choice(["eval", "eval", "step", "step", "step", "adaptive", "adjoint", "rhs",
                       "batch", "targets", "direct"])
    if kind in ("eval", "step"):
        prec = rng.choice(["fp64", "fp32", "fp32", "mixed"])
        top = 1_000_000 if prec == "fp64" else 4_000_000
        c = dict(kind=kind, shape="uniform", n=_logint(rng, 1000, top), **_kappa(rng),
                 p=rng.randint(8, 32 if prec == "fp64" else 24), leaf=rng.choice([16, 24, 32, 48]),
                 prec=prec, grad=rng.random() < 0.75)
        if kind == "step":
            c["wait"] = rng.random() < 0.5
        return c
    if kind == "adaptive":
        return dict(kind=rng.choice(["eval", "step"]), shape="clustered",
                    n=_logint(rng, 20_000, 4_000_000), **_kappa(rng), p=rng.randint(8, 24),
                    leaf=rng.choice([24, 32, 48]), prec=rng.choice(["fp32", "mixed"]), grad=True,
                    wait=True)
    if kind == "adjoint":
        prec = rng.choice(["fp64", "fp32", "fp32"])
        return dict(kind="adjoint", shape="uniform",
                    n=_logint(rng, 2000, 300_000 if prec == "fp64" else 1_000_000), **_kappa(rng),
                    p=rng.randint(10, 24), leaf=rng.choice([32, 48, 64]), prec=prec)
    if kind == "rhs":
        return dict(kind="rhs", shape="uniform", n=_logint(rng, 5000, 500_000), **_kappa(rng),
                    p=rng.randint(8, 20), leaf=rng.choice([24, 32, 48]), prec="fp32",
                    nrhs=rng.randint(2, 64), mode=0)
    if kind == "batch":
        lo = _logint(rng, 1000, 20_000)
        return dict(kind="batch", count=rng.randint(4, 32), lo=lo,
                    hi=_logint(rng, 2 * lo, 400_000), p=rng.randint(8, 20),
                    leaf=rng.choice([24, 32, 48]), prec=rng.choice(["fp32", "fp32", "mixed"]))
    if kind == "targets":
        return dict(kind="targets", per_circle=_logint(rng, 250, 25_000),
                    nfx=rng.randint(64, 500), nfy=rng.randint(31, 250), **_kappa(rng, 2.5),
                    p=rng.randint(10, 24), leaf=rng.randint(3, 16),
                    prec=rng.choice(["fp64", "fp32", "fp32"]))
    nt = _logint(rng, 16, 4096)
    return dict(kind="direct", nt=nt, n=_logint(rng, nt, min(1_000_000, 30_000_000 // nt)),
                **_kappa(rng))


# --------------------------------------------------------------------------
# inputs

# root square (x0, side) that holds the circles and the mesh of ``targets``
CIRCLE_ROOT = (-4.4, 8.8)


def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)


def _points(shape, n, g):
    """Points of [0, 1) x (0, 1]: a uniform cloud, or four fifths of it in 64
    Gaussian clusters (sigma 0.01) with centres next to the boundary y = 0."""
    x, y = _rand(g, n), 1.0 - _rand(g, n)
    if shape == "clustered":
        m = (4 * n) // 5
        cx, cy = _rand(g, 64), 0.001 + 0.049 * (1.0 - _rand(g, 64))
        which = torch.arange(m, device="cuda") % 64
        todo = torch.arange(m, device="cuda")
        while todo.numel():  # a point outside the square is drawn again
            z = torch.randn(2, todo.numel(), dtype=torch.float64, device="cuda", generator=g)
            tx, ty = cx[which[todo]] + 0.01 * z[0], cy[which[todo]] + 0.01 * z[1]
            ok = (tx >= 0) & (tx <= 1) & (ty > 0) & (ty <= 1)
            x[todo[ok]], y[todo[ok]] = tx[ok], ty[ok]
            todo = todo[~ok]
    return x, y


def _charges(g, *shape):
    return 2.0 * _rand(g, *shape) - 1.0


def _batch_problems(case):
    """Sizes log-uniform in [lo, hi] and Robin parameters uniform in [0.1, 10]."""
    g = np.random.Generator(np.random.PCG64(0))
    n = np.floor(10.0 ** g.uniform(math.log10(case["lo"]), math.log10(case["hi"]),
                                   case["count"])).astype(int)
    return [int(k) for k in n], [float(k) for k in g.uniform(0.1, 10.0, case["count"])]


def _circles(case, seed):
    """Eight circles of radius 1, each cut into equal arcs carrying charges, and
    a mesh of field points over them whose bottom row lies on y = 0."""
    g = _rng(seed)
    m = case["per_circle"]
    turn = _rand(g, 8)  # where each circle's cut begins
    k = torch.arange(m, dtype=torch.float64, device="cuda")
    xs, ys = [], []
    for c in range(8):
        th = TWO_PI * (k + turn[c]) / m
        xs.append(-3.3 + 2.2 * (c % 4) + torch.cos(th))
        ys.append((1.01 if c < 4 else 3.2) + torch.sin(th))
    q = TWO_PI / m * (1.0 + 0.5 * _charges(g, 8 * m))
    gx = torch.linspace(-4.4, 4.4, case["nfx"], dtype=torch.float64, device="cuda")
    gy = torch.linspace(0.0, 4.2, case["nfy"], dtype=torch.float64, device="cuda")
    ty, tx = torch.meshgrid(gy, gx, indexing="ij")
    return (torch.cat(xs), torch.cat(ys), q, tx.reshape(-1).contiguous(),
            ty.reshape(-1).contiguous())


def _inputs(case, seed):
    """The inputs of a case, from the seed alone."""
    kind = case["kind"]
    if kind == "batch":
        g = _rng(seed)
        sizes, kappas = _batch_problems(case)
        return [(*_points("uniform", n, g), _charges(g, n), k) for n, k in zip(sizes, kappas)]
    if kind == "targets":
        return _circles(case, seed)
    g = _rng(seed)
    n = case["n"]
    x, y = _points(case.get("shape", "uniform"), n, g)
    q = _charges(g, case["nrhs"], n) if kind == "rhs" else _charges(g, n)
    if kind == "adjoint":
        return x, y, q, _charges(g, n)
    if kind == "direct":
        at = torch.sort(torch.randperm(n, device="cuda", generator=g)[:case["nt"]]).values
        return x, y, q, at
    return x, y, q


# --------------------------------------------------------------------------
# one pass


def _single(case):
    return case.get("prec", "fp64") != "fp64"


def prepare(case, seed):
    kind, ins = case["kind"], _inputs(case, seed)
    kappa = complex(case.get("kre", 1.0), case.get("kim", 0.0))
    s = dict(case=case, kind=kind, ins=ins)
    if kind == "batch":
        plans = [hp.hpfmm_create(x, y, kappa=k, p=case["p"], leaf_size=case["leaf"],
                                 prec=case["prec"]) for x, y, _, k in ins]
        s["batch"] = hp.hpfmm_batch_create(plans)
    elif kind == "targets":
        s["plan"] = hp.hpfmm_create(ins[0], ins[1], kappa=kappa, p=case["p"],
                                    leaf_size=case["leaf"], prec=case["prec"],
                                    root=CIRCLE_ROOT)
    elif kind == "direct":
        x, y, _, at = ins
        s["xt"], s["yt"] = x[at].contiguous(), y[at].contiguous()
    else:
        s["plan"] = hp.hpfmm_create(ins[0], ins[1], kappa=kappa, p=case["p"],
                                    leaf_size=case["leaf"], prec=case["prec"],
                                    adaptive=case["shape"] == "clustered",
                                    m2l_mode=case.get("mode", 0),
                                    async_update=kind == "step" and not case["wait"])
    s["kappa"] = kappa
    return s


def run(state):
    case, kind, ins = state["case"], state["kind"], state["ins"]
    if kind == "eval":
        out = hp.hpfmm_eval(state["plan"], ins[2], grad=case["grad"])
    elif kind == "step":
        hp.hpfmm_update_points(state["plan"], ins[0], ins[1])
        out = hp.hpfmm_eval(state["plan"], ins[2], grad=case["grad"])
    elif kind == "rhs":
        out = hp.hpfmm_eval(state["plan"], ins[2], grad=True)
    elif kind == "adjoint":
        x, y, q = (t.detach().requires_grad_(True) for t in ins[:3])
        u = hp.potential(x, y, q, plan=state["plan"])
        out = (u.detach(), *torch.autograd.grad(u, (x, y, q), ins[3].to(u.dtype)))
    elif kind == "batch":
        pots, grads = hp.hpfmm_eval_batched(state["batch"], [p[2] for p in ins], grad=True)
        # the whole batch as two tensors, problem after problem
        out = (torch.cat(pots), torch.cat(grads))
    elif kind == "targets":
        out = hp.hpfmm_eval_targets(state["plan"], ins[2], ins[3], ins[4], grad=True)
    else:
        out = hp.hpfmm_direct(ins[0], ins[1], ins[2], state["xt"], state["yt"],
                              kappa=state["kappa"], self_index=ins[3], grad=True)
    out = [t for t in out if t is not None]
    if _single(case) and kind != "direct":
        out = [t.to(torch.complex64 if t.is_complex() else torch.float32) for t in out]
    return out


# --------------------------------------------------------------------------
# what one pass cannot do without


def _fmm_work(n, p, leaf, nrhs=1, grad=True):
    """Bytes and operations of one FMM pass set over n points: the charges and
    positions read, the results written; nine leaves of near-field pairs a
    point (13 operations each, 7 of them per charge vector), 27 translations a
    leaf and the expansions formed and evaluated at every point."""
    p1 = p + 1
    pairs = 9.0 * leaf * n * (6 + 7 * nrhs)
    m2l = 27.0 * n / leaf * (4.0 / 3.0) * 8 * p1 * p1 * nrhs
    pts = n * 8.0 * p1 * 4 * nrhs
    return dict(bytes=n * (16.0 + nrhs * (8.0 + (48.0 if grad else 16.0))),
                flops=pairs + m2l + pts)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_fmm_work(n, case["p"], case["leaf"]) for n in _batch_problems(case)[0]]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    if kind == "targets":
        ns, nt = 8 * case["per_circle"], case["nfx"] * case["nfy"]
        w = _fmm_work(ns, case["p"], case["leaf"])
        # the sources' side, then the field points' reads, results and expansions
        return dict(bytes=ns * 24.0 + nt * 64.0, flops=w["flops"] + nt * 32.0 * (case["p"] + 1))
    if kind == "direct":
        # free and image pair (13 operations each) and the reaction pair, about 120
        return dict(bytes=case["n"] * 24.0 + case["nt"] * 72.0,
                    flops=146.0 * case["n"] * case["nt"])
    if kind == "adjoint":
        # the forward with its field, then two transpose passes with theirs
        w = _fmm_work(case["n"], case["p"], case["leaf"])
        return dict(bytes=case["n"] * (24.0 + 16.0 + 16.0 + 24.0), flops=3 * w["flops"])
    return _fmm_work(case["n"], case["p"], case["leaf"], case.get("nrhs", 1),
                     case.get("grad", True))


# --------------------------------------------------------------------------
# the same in 64 bits, by direct summation


def _series_terms(a):
    """Terms of sum a^k / (k k!) until they are below 1e-18 of its largest."""
    k, t, top = 1, a, a
    while k < a or t > 1e-18 * max(top, 1e-3):
        k += 1
        t *= a / k
        top = max(top, t / k)
        if k > 400:
            break
    return k


def _j01(P, amax):
    """J_0(P) = e^{-P} [i pi - Ei(P)] with Ei(P) = gamma + Log P + sum_{k>=1} P^k/(k k!),
    and J_1 = 1 + P J_0."""
    nk = _series_terms(amax)
    c = [1.0 / (k * math.factorial(k)) for k in range(1, nk + 1)]
    S = torch.full_like(P, c[-1])
    for ck in reversed(c[:-1]):
        S = torch.addcmul(torch.tensor(ck, dtype=P.dtype, device=P.device), S, P)
    S.mul_(P)
    S.add_(torch.log(P)).add_(EULER_GAMMA)
    J0 = torch.exp(-P) * (1j * math.pi - S)
    return J0, 1.0 + P * J0


def _direct(xs, ys, Q, xt, yt, self_index, kappa):
    """u (R, T) and grad u (R, T, 2) of the half-plane Robin sum for R charge
    vectors Q (R, N); self_index[t] is the source equal to target t, or None."""
    R, N, T = Q.shape[0], xs.numel(), xt.numel()
    pot = torch.empty(R, T, dtype=torch.complex128, device=xs.device)
    grad = torch.empty(R, T, 2, dtype=torch.complex128, device=xs.device)
    spread = max(float(xs.max() - xt.min()), float(xt.max() - xs.min()))
    amax = abs(kappa) * math.hypot(spread, float(ys.max() + yt.max()))
    rows = max(1, (1 << 22) // N)
    Qt = Q.t().contiguous()

    def times(K):  # (t, N) complex by (N, R) real
        return torch.complex(K.real @ Qt, K.imag @ Qt).t()

    for t0 in range(0, T, rows):
        t1 = min(T, t0 + rows)
        X = xt[t0:t1, None] - xs[None, :]
        D = yt[t0:t1, None] - ys[None, :]
        Y = yt[t0:t1, None] + ys[None, :]
        r2 = X * X + D * D
        if self_index is not None:
            r2[torch.arange(t1 - t0, device=xs.device), self_index[t0:t1]] = math.inf
        R2 = X * X + Y * Y
        lr = torch.log(r2)
        lr[torch.isinf(r2)] = 0.0
        real = 0.5 * (torch.log(R2) - lr)
        sp = torch.complex(Y, -X)
        J0, J1 = _j01(kappa * sp, amax)
        tp = J1 / sp
        if kappa.imag == 0.0:
            # conjugate arguments: only i pi is not conjugated with them
            turn = 2j * math.pi * torch.exp(-kappa * sp.conj())
            J0m = J0.conj() + turn
            tm = (1.0 + (kappa * sp.conj()) * J0m) / sp.conj()
        else:
            J0m, J1m = _j01(kappa * sp.conj(), amax)
            tm = J1m / sp.conj()
        pot[:, t0:t1] = times(real + J0 + J0m) / TWO_PI
        grad[:, t0:t1, 0] = times(X / R2 - X / r2 + 1j * (tp - tm)) / TWO_PI
        grad[:, t0:t1, 1] = times(Y / R2 - D / r2 - (tp + tm)) / TWO_PI
    return pot, grad


def _cost(pairs, kappa, reach):
    return pairs * _series_terms(abs(kappa) * reach) * (1 if kappa.imag == 0.0 else 2)


def exact(case, seed):
    kind = case["kind"]
    kappa = complex(case.get("kre", 1.0), case.get("kim", 0.0))
    reach = math.sqrt(5.0)
    if kind == "batch":
        # the problems lie one after the other in the outputs: all or none of them
        sizes, kappas = _batch_problems(case)
        if sum(_cost(float(n) * n, complex(k), reach) for n, k in zip(sizes, kappas)) > EXACT_BUDGET:
            return None
        parts = []
        for x, y, q, k in _inputs(case, seed):
            u, g = _direct(x, y, q[None], x, y, torch.arange(x.numel(), device=x.device), complex(k))
            parts.append((u[0], g[0]))
        return [torch.cat([u for u, _ in parts]), torch.cat([g for _, g in parts])]
    if kind == "targets":
        ns, nt = 8.0 * case["per_circle"], float(case["nfx"] * case["nfy"])
        if _cost(ns * nt, kappa, 12.0) > EXACT_BUDGET:
            return None
        x, y, q, xt, yt = _inputs(case, seed)
        u, g = _direct(x, y, q[None], xt, yt, None, kappa)
        return [u[0], g[0]]
    n = float(case["n"])
    if _cost(n * (case["nt"] if kind == "direct" else n), kappa, reach) > EXACT_BUDGET:
        return None
    ins = _inputs(case, seed)
    x, y, q = ins[:3]
    every = torch.arange(x.numel(), device=x.device)
    if kind == "direct":
        at = ins[3]
        u, g = _direct(x, y, q[None], x[at], y[at], at, kappa)
        return [u[0], g[0]]
    if kind == "rhs":
        return list(_direct(x, y, q, x, y, every, kappa))
    if kind == "adjoint":
        # the kernel is symmetric: the transpose sums are the sums with charges w
        w = ins[3]
        u, g = _direct(x, y, torch.stack([q, w]), x, y, every, kappa)
        d = w[:, None] * g[0].real + q[:, None] * g[1].real
        return [u[0], d[:, 0], d[:, 1], u[1].real]
    u, g = _direct(x, y, q[None], x, y, every, kappa)
    return [u[0], g[0]] if case["grad"] else [u[0]]
