"""Performance cases of the library: what its users have it do, through the public entry points.

Three kinds of call are covered:

* ``eval``   one ``InlaModel.value_and_grad`` call, for one theta or for a set of candidate thetas
             evaluated together (the L-BFGS line search), with or without the gradient, in each
             precision mode, keeping both factors or in the low-memory variant;
* ``batch``  one ``InlaBatch.value_and_grad`` call over several models of uneven block size;
* ``blocks`` the building blocks a program strings together itself: assemble Q_c, factor it with the
             lower solve, solve for the mode, selected inversion with the fused traces.

Sizes are those of the repository's synthetic workloads (cut in the number of time blocks where the
whole model would take seconds a call: every time block costs the same) and ragged ones in between.
A case's inputs (observation design, covariates, observations, theta) are drawn from its seed.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

import paper_2605_06392_gb300 as P


# ---- the cases -----------------------------------------------------------------------------------

def _eval(name, k, nx, ny, nt, a, n_obs, precision, grad=True, thetas=1, low_memory=False, mode=False):
    return dict(name=name, kind="eval", k=k, nx=nx, ny=ny, nt=nt, a=a, n_obs=n_obs, precision=precision,
                grad=grad, thetas=thetas, low_memory=low_memory, mode=mode)


def listed():
    return [
        # the smallest model (8 x 8 grid, 4 steps): one gradient of a quick interactive fit; launches count
        _eval("tiny_f64_grad", 1, 8, 8, 4, 4, 512, 0),
        # three small coregionalised responses (b = 192), one gradient in emulated FP64
        _eval("coreg_small_emu_grad", 3, 8, 8, 5, 9, 3000, 2),
        # an L-BFGS line search: four candidate thetas together, two responses on a ragged 13 x 11 grid
        _eval("line_search_f64", 2, 13, 11, 10, 4, 4000, 0, thetas=4),
        # the medium univariate model (32 x 32 grid) in plain FP64, as the default precision gives it
        _eval("medium_f64_grad", 1, 32, 32, 6, 6, 12_500, 0, mode=True),
        # the same at its full 50 steps in the two tensor-core modes
        _eval("medium_emu_grad", 1, 32, 32, 50, 6, 100_000, 2, mode=True),
        _eval("medium_mixed_grad", 1, 32, 32, 50, 6, 100_000, 1, mode=True),
        # one value-only evaluation of it: a finite-difference or profile-likelihood point
        _eval("medium_emu_value", 1, 32, 32, 50, 6, 100_000, 2, grad=False),
        # the large univariate model (45 x 45 grid: b = 2025 is ragged), emulated FP64
        _eval("large_emu_grad", 1, 45, 45, 16, 8, 64_000, 2, mode=True),
        # the production model (3 x 40 x 40 grid, b = 4800, d = 15), the benchmark's headline call
        _eval("production_emu_grad", 3, 40, 40, 8, 12, 83_334, 2, mode=True),
        # the same when memory is short: off-diagonal factors recomputed
        _eval("production_lowmem_emu", 3, 40, 40, 5, 12, 52_000, 2, low_memory=True),
        # six coregionalised models of uneven size (b = 768, 1728, 3072) in one call
        dict(name="batch_emu_grad", kind="batch", k=3, sides="16,24,32,16,24,16", nt=5, a=9, n_obs=6250,
             precision=2, grad=True),
        # a program that factors, solves and inverts Q_c itself (b = 588, ragged)
        dict(name="blocks_emu", kind="blocks", k=3, nx=14, ny=14, nt=8, a=9, n_obs=5000, precision=2),
    ]


def _shape(rng, k, lo, hi):
    """A ragged grid whose block size k nx ny is log-uniform in lo .. hi."""
    b = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    side = math.sqrt(b / k)
    nx = max(2, round(side * rng.uniform(0.8, 1.25)))
    return nx, max(2, min(round(b / k / nx), int(hi / k / nx)))


def _seconds(b, nt, precision, grad, thetas=1):
    """A rough upper estimate of one pass, to keep a drawn case below the largest listed one."""
    fl = _flops(b, nt, grad) * thetas
    return fl / 1.0e12 if precision == 0 else fl / 2.5e13 + thetas * nt * (b / 32) * 60e-6


def draw(rng):
    u = rng.random()
    if u < 0.1:
        sides = [str(rng.randint(10, 28)) for _ in range(rng.randint(2, 6))]
        return dict(kind="batch", k=3, sides=",".join(sides), nt=rng.randint(3, 6), a=9,
                    n_obs=rng.randint(2000, 8000), precision=rng.choice([1, 2, 2]), grad=rng.random() < 0.8)
    if u < 0.2:
        k = rng.randint(1, 3)
        nx, ny = _shape(rng, k, 100, 700)
        return dict(kind="blocks", k=k, nx=nx, ny=ny, nt=rng.randint(3, 9), a=3 * k, n_obs=rng.randint(1000, 6000),
                    precision=rng.choice([0, 2, 2]))
    k = rng.choice([1, 1, 2, 3])
    precision = rng.choice([0, 1, 2, 2, 2])
    grad = rng.random() < 0.75
    nx, ny = _shape(rng, k, 48, 1100 if precision == 0 else 4800)
    b = k * nx * ny
    thetas = 4 if b <= 600 and rng.random() < 0.3 else 1
    nt = round(math.exp(rng.uniform(math.log(2), math.log(60))))
    while nt > 2 and _seconds(b, nt, precision, grad, thetas) > 0.3:
        nt -= 1
    return dict(kind="eval", k=k, nx=nx, ny=ny, nt=nt, a=k * rng.randint(1, 4), n_obs=rng.randint(500, 2000) * nt,
                precision=precision, grad=grad, thetas=thetas,
                low_memory=precision != 1 and rng.random() < 0.15, mode=rng.random() < 0.5)


# ---- inputs --------------------------------------------------------------------------------------

def _problem(k, nx, ny, nt, a, n_obs, rng):
    """Observations of a smooth space-time field plus fixed effects and noise, and thetas near the
    ones that generated them."""
    ns, a_r = nx * ny, a // k
    obs_v = (np.arange(n_obs) % k).astype(np.int32)
    rng.shuffle(obs_v)
    obs_t = rng.integers(0, nt, n_obs).astype(np.int32)
    obs_s = rng.integers(0, ns, n_obs).astype(np.int32)
    cov = rng.standard_normal((n_obs, a_r))
    if k == 1:
        true = np.array([0.3, 1.0, -0.5, 1.5])
    else:
        true = np.concatenate([np.full(k, 0.4), np.full(k, -0.3), np.zeros(k),
                               np.full(k * (k - 1) // 2, 0.3), np.full(k, 1.5)])
        cov[:, 0] = 1.0
    beta = rng.standard_normal((k, a_r))
    w = rng.integers(0, 3, (8, 3)) * (2 * math.pi / np.array([nt, ny, nx]))
    amp, ph = rng.standard_normal((k, 8)) / math.sqrt(8), rng.uniform(0, 2 * math.pi, 8)
    at = np.stack([obs_t, obs_s // nx, obs_s % nx], axis=1).astype(np.float64)
    field = np.einsum("nm,nm->n", np.sin(at @ w.T + ph), amp[obs_v])
    noise = rng.standard_normal(n_obs) * math.exp(-0.75)
    y = field + np.einsum("nc,nc->n", cov, beta[obs_v]) + noise
    prob = types.SimpleNamespace(k=k, nx=nx, ny=ny, ns=ns, b=k * ns, nt=nt, a=a, a_r=a_r, obs_t=obs_t,
                                 obs_s=obs_s, obs_v=obs_v, obs_cov=cov, y=y)
    return prob, true


def _inputs(case, seed):
    """[(problem, thetas)] of a case: one entry per model."""
    rng = np.random.default_rng(seed)
    grids = [(int(s), int(s)) for s in case["sides"].split(",")] if case["kind"] == "batch" \
        else [(case["nx"], case["ny"])]
    got = []
    for nx, ny in grids:
        prob, true = _problem(case["k"], nx, ny, case["nt"], case["a"], case["n_obs"], rng)
        th = true + 0.1 * rng.standard_normal(true.shape)
        if case.get("thetas", 1) > 1:      # step lengths along one search direction
            p = rng.standard_normal(true.shape) * 0.05
            th = np.array([th + t * p for t in (1.0, 0.5, 0.25, 0.1)])
        got.append((prob, th))
    return got


def prepare(case, seed):
    inputs = _inputs(case, seed)
    models = [P.InlaModel(p, low_memory=case.get("low_memory", False)) for p, _ in inputs]
    s = types.SimpleNamespace(case=case, models=models, model=models[0], theta=inputs[0][1],
                              thetas=[t for _, t in inputs])
    if case["kind"] == "batch":
        s.batch = P.InlaBatch(models)
    if case["kind"] == "blocks":
        m = s.model
        s.q = m.new_matrix(1)
        s.x = torch.empty(m.n * m.ld + m.a, dtype=torch.float64, device="cuda")
    return s


def run(s):
    c = s.case
    if c["kind"] == "batch":
        f, grads = s.batch.value_and_grad(s.thetas, grad=c["grad"], precision=c["precision"])
        return {"f": f, "grad": grads}
    if c["kind"] == "blocks":
        P.bta_assemble(s.model, s.theta, 1, s.q, rhs=s.x)
        logdet, fail = P.bta_factor(s.q, rhs=s.x, precision=c["precision"])
        P.bta_solve(s.q, s.x)
        traces = P.bta_selinv(s.q, s.model, s.theta, 1)
        return {"logdet": logdet, "fail": fail, "x": s.x, "traces": traces, "D": s.q.D, "B": s.q.B,
                "C": s.q.C, "T": s.q.T}
    f, g = s.model.value_and_grad(s.theta, grad=c["grad"], concurrent=c["thetas"], precision=c["precision"])
    return {"f": f, "grad": g, "mode": s.model.mode() if c["mode"] else None}


# ---- work ----------------------------------------------------------------------------------------

def _flops(b, nt, grad):
    """Block Cholesky with the inverse diagonal factors (8/3 b^3 a block) and the selected inversion
    (13/3 b^3) of Q_c and Q_p, triangles and symmetry used."""
    return 2.0 * nt * b ** 3 * (8 / 3 + (13 / 3 if grad else 0.0))


def work(case):
    """Bytes: a call has the model's stencils, observations and thetas to read and f, the gradient
    (and x*) to write; the building blocks also write their matrix."""
    n = len(case["sides"].split(",")) if case["kind"] == "batch" else 1
    per_obs = 8.0 * (case["a"] // case["k"] + 1) + 12
    if case["kind"] == "batch":
        fl = sum(_flops(3 * int(s) ** 2, case["nt"], case["grad"]) for s in case["sides"].split(","))
        return {"bytes": n * case["n_obs"] * per_obs, "flops": fl}
    b, nt = case["k"] * case["nx"] * case["ny"], case["nt"]
    byt = case["n_obs"] * per_obs + 8.0 * nt * b
    if case["kind"] == "blocks":
        return {"bytes": byt + 8.0 * (2 * nt - 1) * b * b, "flops": _flops(b, nt, True) / 2}
    return {"bytes": byt * case["thetas"], "flops": _flops(b, nt, case["grad"]) * case["thetas"]}


# ---- the same results from plain 64-bit torch ------------------------------------------------------
# Q_p = sum_j Mj (x) sum_s coef[j][p][q][s] S_s on blocks of time steps, Q_c = Q_p + A^T tau A.

def _coefs(th, k):
    """coef[j, p, q, s] (temporal matrix j, responses p and q, spatial matrix s) and tau from theta."""
    one, zero = torch.ones_like(th[0]), torch.zeros_like(th[0])

    def unit(kap, gam):
        return torch.stack([torch.stack([kap ** 4, 2 * kap ** 2, one]),
                            torch.stack([2 * kap ** 3 * gam, 2 * kap * gam, zero]),
                            torch.stack([one, zero, zero])])

    if k == 1:
        u = torch.exp(th[0]) * unit(torch.exp(th[1]), torch.exp(th[2]))
        return u[:, None, None, :], torch.exp(th[3:4])
    lam = torch.diag(torch.exp(th[2 * k:3 * k]))
    low = torch.tril_indices(k, k, -1, device=th.device)
    lam = lam.index_put((low[0], low[1]), th[3 * k:3 * k + low.shape[1]])
    li = torch.linalg.inv(lam)
    u = torch.stack([unit(torch.exp(th[m]), torch.exp(th[k + m])) for m in range(k)])
    return torch.einsum("mp,mq,mjs->jpqs", li, li, u), torch.exp(th[-k:])


def _logdet_prior(th, prob):
    """log|Q_st| from the spectra of the grid Laplacian and of tridiag(-1, 2, -1)."""
    k, dev = prob.k, th.device

    def lap(m):
        return 2 - 2 * torch.cos(math.pi * torch.arange(m, dtype=torch.float64, device=dev) / m)

    g = (lap(prob.ny)[:, None] + lap(prob.nx)[None, :]).reshape(-1)[None, :]
    t = torch.arange(1, prob.nt + 1, dtype=torch.float64, device=dev)
    m1 = (2 - 2 * torch.cos(math.pi * t / (prob.nt + 1)))[:, None]
    ld = 0.0
    for m in range(k):
        kap, gam = (torch.exp(th[1]), torch.exp(th[2])) if k == 1 else (torch.exp(th[m]), torch.exp(th[k + m]))
        k0, k1 = kap ** 4 + 2 * kap ** 2 * g + g * g, kap ** 2 + g
        ld = ld + torch.log(k0 + 2 * kap * gam * m1 * k1 + 1).sum()
    n = prob.nt * prob.ns
    return ld + n * th[0] if k == 1 else ld - 2 * n * th[2 * k:3 * k].sum()


def _exact_one(prob, theta, grad=True, inverse=False):
    """f, its gradient, x*, and on request log|Q_c|, the traces and the selected inverse of Q_c."""
    dev, f64 = "cuda", torch.float64
    k, nt, ns, b, a, a_r = prob.k, prob.nt, prob.ns, prob.b, prob.a, prob.a_r
    th = torch.tensor(theta, dtype=f64, device=dev, requires_grad=True)
    coef, tau = _coefs(th, k)
    cf, tu = coef.detach(), tau.detach()
    one_d = [torch.diag(torch.full((m,), 2.0, dtype=f64, device=dev)) for m in (prob.nx, prob.ny)]
    for d in one_d:
        m = d.shape[0]
        d -= torch.diag(torch.ones(m - 1, dtype=f64, device=dev), 1) + torch.diag(torch.ones(m - 1, dtype=f64, device=dev), -1)
        d[0, 0] -= 1
        d[-1, -1] -= 1
    eye = [torch.eye(m, dtype=f64, device=dev) for m in (prob.nx, prob.ny)]
    G = torch.kron(eye[1], one_d[0]) + torch.kron(one_d[1], eye[0])
    S = torch.stack([torch.eye(ns, dtype=f64, device=dev), G, G @ G])

    def spread(w):   # [p, q, s] -> the b x b block
        return torch.einsum("pqs,sij->piqj", w, S).reshape(b, b)

    D0, B0 = spread(cf[0] + 2 * cf[1] + cf[2]), spread(-cf[1])
    # A^T A pieces, per response
    o_t, o_v = (torch.from_numpy(x.astype(np.int64)).to(dev) for x in (prob.obs_t, prob.obs_v))
    lat = o_t * b + o_v * ns + torch.from_numpy(prob.obs_s.astype(np.int64)).to(dev)
    y = torch.from_numpy(prob.y).to(dev)
    cov = torch.zeros(len(y), a, dtype=f64, device=dev)
    fe = o_v[:, None] * a_r + torch.arange(a_r, device=dev)[None, :]
    cov.scatter_(1, fe, torch.from_numpy(prob.obs_cov).to(dev))
    w = tu[o_v]
    cnt = torch.zeros(nt * b, dtype=f64, device=dev).index_add_(0, lat, torch.ones_like(y))
    tau_lat = tu.repeat_interleave(ns).repeat(nt)
    C0 = torch.zeros(nt * b, a, dtype=f64, device=dev).index_add_(0, lat, cov)   # A_lat^T A_fe, unscaled
    tau_fe = tu.repeat_interleave(a_r)
    T0 = 1e-3 * torch.eye(a, dtype=f64, device=dev) + cov.T @ (w[:, None] * cov)
    r = torch.cat([torch.zeros(nt * b, dtype=f64, device=dev).index_add_(0, lat, w * y), cov.T @ (w * y)])
    C = [(C0[t * b:(t + 1) * b] * tau_fe).T for t in range(nt)]
    # block Cholesky of Q_c with the lower solve
    tri = torch.linalg.solve_triangular
    L, LB, LC, z, logdet, T, D, rT = [], [], [], [], 0.0, T0, None, r[nt * b:].clone()
    for t in range(nt):
        D = D0 + torch.diag((tau_lat * cnt)[t * b:(t + 1) * b])
        rt, Ct = r[t * b:(t + 1) * b], C[t]
        if t:
            D, rt, Ct = D - LB[-1] @ LB[-1].T, rt - LB[-1] @ z[-1], Ct - LC[-1] @ LB[-1].T
        L.append(torch.linalg.cholesky(D))
        logdet = logdet + 2 * torch.log(torch.diagonal(L[t])).sum()
        z.append(tri(L[t], rt[:, None], upper=False)[:, 0])
        LC.append(tri(L[t], Ct.T, upper=False).T)
        T, rT = T - LC[t] @ LC[t].T, rT - LC[t] @ z[t]
        if t < nt - 1:
            LB.append(tri(L[t], B0.T, upper=False).T)
    LT = torch.linalg.cholesky(T)
    logdet = logdet + 2 * torch.log(torch.diagonal(LT)).sum()
    xT = torch.cholesky_solve(rT[:, None], LT)[:, 0]
    x = [None] * nt
    for t in range(nt - 1, -1, -1):
        v = z[t] - LC[t].T @ xT
        if t < nt - 1:
            v = v - LB[t].T @ x[t + 1]
        x[t] = tri(L[t].T, v[:, None], upper=True)[:, 0]
    X = torch.stack(x)
    # f of Eq. 1 with its quadratic form and likelihood as functions of theta at fixed x*
    Xk = X.reshape(nt, k, ns)
    SX = torch.einsum("sij,tqj->stqi", S, Xk)
    same = torch.einsum("tpi,stqi->tpqs", Xk, SX).sum(0)
    nxt = torch.einsum("tpi,stqi->pqs", Xk[1:], SX[:, :-1])
    nxt = nxt + nxt.transpose(0, 1)
    RX = torch.stack([same, 2 * same - nxt, same])
    res = y - X.reshape(-1)[lat] - cov @ xT
    rs = torch.zeros(k, dtype=f64, device=dev).index_add_(0, o_v, res * res)
    nv = torch.bincount(o_v, minlength=k).to(f64)
    quad = (coef * RX).sum() + 1e-3 * (xT @ xT)
    rest = 0.5 * _logdet_prior(th, prob) + 0.5 * a * math.log(1e-3) - 0.5 * quad \
        + (0.5 * nv * torch.log(tau) - 0.5 * tau * rs).sum() - (th @ th) / 200.0
    f = float(rest.detach()) - 0.5 * float(logdet)
    out = {"f": f, "x": torch.cat([X.reshape(-1), xT]), "logdet": logdet}
    if not grad:
        return out
    # selected inversion of Q_c, contracted with the stencils
    ZT = torch.cholesky_inverse(LT)
    R = torch.zeros_like(RX)
    tc = torch.zeros(k, dtype=f64, device=dev)
    tc = tc + torch.diagonal(ZT @ (cov.T @ cov)).reshape(k, a_r).sum(1)
    ZD = ZC = None
    blocks = []
    for t in range(nt - 1, -1, -1):
        li = tri(L[t], torch.eye(b, dtype=f64, device=dev), upper=False)
        FC = LC[t] @ li
        nC = -ZT @ FC
        ZB = None
        if t < nt - 1:
            FB = LB[t] @ li
            nC = nC - ZC @ FB
            ZB = -ZD @ FB - ZC.T @ FC
        ZD = li.T @ li - nC.T @ FC
        if ZB is not None:
            ZD = ZD - ZB.T @ FB
            R[1] -= 2 * torch.einsum("piqj,sij->pqs", ZB.reshape(k, ns, k, ns), S)
        dd = torch.einsum("piqj,sij->pqs", ZD.reshape(k, ns, k, ns), S)
        R += torch.stack([dd, 2 * dd, dd])
        ZC = nC
        tc = tc + (torch.diagonal(ZD) * cnt[t * b:(t + 1) * b]).reshape(k, ns).sum(1)
        tc = tc + 2 * (ZC * C0[t * b:(t + 1) * b].T).sum(1).reshape(k, a_r).sum(1)
        if inverse:
            blocks.append((ZD, ZB, ZC))
    trace = (coef * R).sum() + (tau * tc).sum()
    out["traces"] = torch.autograd.grad(trace, th, retain_graph=True)[0]
    out["grad"] = torch.autograd.grad(rest, th)[0] - 0.5 * out["traces"]
    out["Z"], out["ZT"] = blocks[::-1], ZT
    return out


def exact(case, seed):
    inputs = _inputs(case, seed)
    if case["kind"] == "batch":
        e = [_exact_one(p, t, case["grad"]) for p, t in inputs]
        return {"f": np.array([v["f"] for v in e]),
                "grad": [v["grad"].cpu().numpy() for v in e] if case["grad"] else None}
    prob, theta = inputs[0]
    if case["kind"] == "blocks":
        e = _exact_one(prob, theta, inverse=True)
        b, nt, a = prob.b, prob.nt, prob.a
        ld = (b + 31) // 32 * 32
        D = torch.eye(ld, dtype=torch.float64, device="cuda").repeat(nt, 1, 1)
        B = torch.zeros(max(nt - 1, 1), ld, ld, dtype=torch.float64, device="cuda")
        C = torch.zeros(nt, ld, a, dtype=torch.float64, device="cuda")
        x = torch.zeros(nt, ld, dtype=torch.float64, device="cuda")
        x[:, :b] = e["x"][:nt * b].reshape(nt, b)
        for t, (zd, zb, zc) in enumerate(e["Z"]):
            D[t, :b, :b] = zd.T
            C[t, :b] = zc.T
            if zb is not None:
                B[t, :b, :b] = zb.T
        return {"logdet": e["logdet"].reshape(1), "fail": None, "x": torch.cat([x.reshape(-1), e["x"][nt * b:]]),
                "traces": e["traces"], "D": D, "B": B, "C": C, "T": e["ZT"]}
    many = np.atleast_2d(theta)
    e = [_exact_one(prob, t, case["grad"]) for t in many]
    f = np.array([v["f"] for v in e])
    g = np.stack([v["grad"].cpu().numpy() for v in e]) if case["grad"] else None
    if np.ndim(theta) == 1:
        f, g = f[0], g[0] if case["grad"] else None
    # x* of a set of thetas is that of its first
    return {"f": f, "grad": g, "mode": e[0]["x"] if case["mode"] else None}
