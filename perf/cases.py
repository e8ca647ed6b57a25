"""The work that users of this library have it do, as cases that can be timed.

Every case goes through the public entry points: the calls of include/eot.h as
the Python package binds them, and the autograd function on top of them. A case
is one call, or the few calls that make one step of a user's program:

  marginals    the plan's marginals at given potentials (a convergence check)
  hvp          one Hessian-vector product of the dual (an outer second-order method)
  backward     the gradients at potentials that the program already has
  match        the plan's integer outputs: each row's best partner and the support
  round        the feasible plan after a solve, with its transport cost
  solve        one full solve to potentials
  train        value and gradients by the autograd function (solve, value, backward)
  batch        many small point problems solved in one launch, then their gradients

Sizes, costs, weights and temperatures are those of this repository's workloads
(image grids, uniform points, colour clouds, high-dimensional mixtures) and the
range around them. Inputs come from the seed alone, in plain torch.
"""
import math

import numpy as np
import torch

import paper_2504_02067_gb300 as E

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the 28 x 28 image grid in double precision: the smallest call in earnest, a
        # convergence check after each step of a user's own scheme
        dict(name="marginals_f64_grid28", op="marginals", cost="grid", prec="fp64", n=784, m=784, kind="sqeuclid",
             gamma=4096.0),
        # a general double-precision cost of odd size (rows not 16-byte aligned)
        dict(name="hvp_f64_1501x1999", op="hvp", cost="dense", prec="fp64", n=1501, m=1999, gamma=1024.0),
        # the 64 x 64 image grid, the benchmark's own size
        dict(name="hvp_mixed_grid64", op="hvp", cost="grid", prec="mixed", n=4096, m=4096, kind="sqeuclid",
             gamma=16384.0),
        # the full method in double precision on the 28 x 28 grid
        dict(name="solve_f64_grid28", op="solve", cost="grid", prec="fp64", n=784, m=784, kind="sqeuclid",
             gamma=4096.0),
        # a learned dense cost: one training step on the 64 x 64 grid (the benchmark's workload)
        dict(name="train_mixed_grid64", op="train", cost="grid", prec="mixed", n=4096, m=4096, kind="sqeuclid",
             gamma=16384.0),
        # moving a small planar point set: one training step
        dict(name="train_points_d2_1000x700", op="train", cost="points", prec="mixed", n=1000, m=700, d=2,
             gamma=1024.0),
        # high-dimensional embeddings (the d = 64 mixtures): one training step
        dict(name="train_points_d64_16384", op="train", cost="points", prec="mixed", n=16384, m=16384, d=64,
             gamma=1024.0),
        # colour transfer: the displacement of every colour at the potentials of the last solve
        dict(name="backward_points_d3_65536", op="backward", cost="points", prec="mixed", n=65536, m=65536, d=3,
             gamma=1024.0),
        # assignments read off the plan of embeddings
        dict(name="match_points_d64_8192", op="match", cost="points", prec="mixed", n=8192, m=8192, d=64,
             gamma=1024.0),
        # assignments on the 64 x 64 grid
        dict(name="match_grid64", op="match", cost="grid", prec="mixed", n=4096, m=4096, kind="l1", gamma=16384.0),
        # the feasible plan of the 64 x 64 grid
        dict(name="round_grid64", op="round", cost="grid", prec="mixed", n=4096, m=4096, kind="sqeuclid",
             gamma=16384.0),
        # many small planar problems of uneven size, trained together
        dict(name="batch_points_d2_48", op="batch", cost="points", prec="mixed", count=48, lo=256, hi=1024, d=2,
             gamma=1024.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["marginals", "hvp", "backward", "match", "round", "solve", "train", "train", "batch"])
    g = lambda lo, hi: float(2 ** rng.randint(lo, hi))  # noqa: E731
    if op == "solve":
        s = rng.randint(12, 28)
        return dict(op=op, cost="grid", prec="fp64", n=s * s, m=s * s, kind="sqeuclid", gamma=g(8, 12))
    if op == "batch":
        lo = _log_int(rng, 64, 400)
        return dict(op=op, cost="points", prec="mixed", count=rng.randint(8, 48), lo=lo, hi=rng.randint(lo, 1024),
                    d=rng.randint(1, 4), gamma=g(8, 10))
    if op == "train":
        if rng.random() < 0.3:
            s = rng.randint(24, 64)
            return dict(op=op, cost="grid", prec="mixed", n=s * s, m=s * s, kind="sqeuclid", gamma=g(10, 14))
        d = rng.choice([2, 3, 4, 7, 16, 17, 24, 32, 48, 64])
        hi = 3000 if d <= 16 else 10000
        return dict(op=op, cost="points", prec="mixed", n=_log_int(rng, 500, hi), m=_log_int(rng, 500, hi), d=d,
                    gamma=g(8, 10))
    if op == "backward":
        if rng.random() < 0.25:
            return dict(op=op, cost="dense", prec="mixed", n=_log_int(rng, 200, 8000), m=_log_int(rng, 200, 8000),
                        gamma=g(8, 12))
        d = rng.choice([1, 2, 3, 5, 8, 16, 33, 64])
        hi = 65536 if d <= 4 else 16384
        return dict(op=op, cost="points", prec="mixed", n=_log_int(rng, 300, hi), m=_log_int(rng, 300, hi), d=d,
                    gamma=g(8, 12))
    if op == "match":
        if rng.random() < 0.5:
            s = rng.randint(20, 80)
            return dict(op=op, cost="grid", prec="mixed", n=s * s, m=s * s, kind=rng.choice(["sqeuclid", "l1"]),
                        gamma=g(10, 14))
        return dict(op=op, cost="points", prec="mixed", n=_log_int(rng, 300, 10000), m=_log_int(rng, 300, 10000),
                    d=rng.choice([1, 2, 3, 8, 20, 64]), gamma=g(8, 12))
    if op == "round":
        if rng.random() < 0.4:
            return dict(op=op, cost="points", prec="mixed", n=_log_int(rng, 300, 6000), m=_log_int(rng, 300, 6000),
                        d=rng.choice([2, 3, 8]), gamma=g(8, 12))
        s = rng.randint(20, 64)
        return dict(op=op, cost="grid", prec=rng.choice(["mixed", "fp64"]), n=s * s, m=s * s,
                    kind=rng.choice(["sqeuclid", "l1"]), gamma=g(10, 14))
    # marginals and Hessian-vector products
    if rng.random() < 0.3:
        return dict(op=op, cost="points", prec="fp64", n=_log_int(rng, 100, 3000), m=_log_int(rng, 100, 3000),
                    d=rng.choice([2, 3, 8, 20]), gamma=g(6, 12))
    return dict(op=op, cost="dense", prec="mixed" if op == "hvp" and rng.random() < 0.5 else "fp64",
                n=_log_int(rng, 100, 4096), m=_log_int(rng, 100, 4096), gamma=g(6, 12))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _grid_cost(side, kind):
    """Squared-Euclidean or L1 cost between the pixel centres of a side x side grid, max 1."""
    a = torch.arange(side, dtype=F64, device=DEV)
    x, y = a.repeat_interleave(side), a.repeat(side)
    dx, dy = x[:, None] - x[None, :], y[:, None] - y[None, :]
    C = dx * dx + dy * dy if kind == "sqeuclid" else dx.abs() + dy.abs()
    return C / C.max()


def _histogram(rng, side, zeros):
    """Three isotropic Gaussians on the grid; `zeros` of the bins empty, else a small floor."""
    a, b = np.meshgrid(np.arange(side), np.arange(side), indexing="ij")
    h = np.zeros((side, side))
    for _ in range(3):
        ca, cb = rng.uniform(0, side, size=2)
        s = rng.uniform(4.0, 12.0) * side / 64
        h += rng.uniform(0.2, 1.0) * np.exp(-0.5 * ((a - ca) ** 2 + (b - cb) ** 2) / s ** 2)
    h = h.ravel()
    if zeros:
        h[rng.choice(h.size, size=int(round(zeros * h.size)), replace=False)] = 0.0
    else:
        h += 1e-6
    return torch.tensor(h / h.sum(), device=DEV)


def _weights(gen, n, uniform):
    if uniform:
        return torch.full((n,), 1.0 / n, dtype=F64, device=DEV)
    w = -torch.log(torch.rand(n, generator=gen, dtype=F64, device=DEV).clamp_min(1e-12))  # Dirichlet(1)
    return w / w.sum()


def _cloud(gen, n, d):
    """d <= 2: uniform in the unit cube; d = 3, 4: colours (16 narrow clusters, clipped to
    the cube); above: eight unit Gaussians with means N(0, 4 I)."""
    if d <= 2:
        return torch.rand(n, d, generator=gen, device=DEV)
    k = 16 if d <= 4 else 8
    if d <= 4:
        means = 0.1 + 0.8 * torch.rand(k, d, generator=gen, device=DEV)
        width = 0.02 + 0.08 * torch.rand(k, 1, generator=gen, device=DEV)
    else:
        means = 2.0 * torch.randn(k, d, generator=gen, device=DEV)
        width = torch.ones(k, 1, device=DEV)
    at = torch.randint(0, k, (n,), generator=gen, device=DEV)
    x = means[at] + width[at] * torch.randn(n, d, generator=gen, device=DEV)
    return (x.clamp(0.0, 1.0) if d <= 4 else x).contiguous()


def _make(case, seed):
    """(C or None, X, Y, r, c, scale): the problem's data."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 1000003 + 17)
    rng = np.random.Generator(np.random.PCG64(int(seed) + 101))
    n, m = case["n"], case["m"]
    if case["cost"] == "grid":
        side = int(round(math.sqrt(n)))
        C = _grid_cost(side, case["kind"])
        zeros = 0.0 if case["prec"] == "fp64" else 0.10
        r, c = _histogram(rng, side, zeros), _histogram(rng, side, zeros)
        return (C if case["prec"] == "fp64" else C.float()), None, None, r, c, 0.0
    if case["cost"] == "dense":
        C = torch.rand(n, m, generator=gen, dtype=F64, device=DEV)
        r, c = _weights(gen, n, False), _weights(gen, m, False)
        return (C if case["prec"] == "fp64" else C.float()), None, None, r, c, 0.0
    d = case["d"]
    X, Y = _cloud(gen, n, d), _cloud(gen, m, d)
    r, c = _weights(gen, n, d > 2), _weights(gen, m, d > 2)
    # the squared diagonal of the clouds' common box bounds the largest squared distance
    lo, hi = torch.minimum(X.amin(0), Y.amin(0)), torch.maximum(X.amax(0), Y.amax(0))
    scale = 1.0 / float(((hi - lo).double() ** 2).sum())
    return None, X, Y, r, c, scale


def _lse_rows(off, C, X, Y, gamma, scale):
    """log sum_j exp(off_j - gamma C_ij) for every row, in blocks of rows."""
    if C is not None:
        return torch.logsumexp(off[None, :] - gamma * C, dim=1)
    out = torch.empty(X.shape[0], dtype=F64, device=DEV)
    step = max(1, (1 << 27) // Y.shape[0])
    o32, yy = off.float(), (Y * Y).sum(1)
    for i in range(0, X.shape[0], step):
        x = X[i:i + step]
        D = ((x * x).sum(1)[:, None] + yy[None, :] - 2.0 * (x @ Y.T)).clamp_min(0.0)
        out[i:i + step] = torch.logsumexp(o32[None, :] - (gamma * scale) * D, dim=1).double()
    return out


def _potentials(C, X, Y, r, c, gamma, scale):
    """Potentials that a program has in hand near the end of its own scheme: a few
    Sinkhorn steps along a rising gamma, on slightly smoothed marginals."""
    C = None if C is None else C.double()
    Ct = None if C is None else C.T
    logr = torch.log(r * (1 - 1e-5) + 1e-5 / r.numel())
    logc = torch.log(c * (1 - 1e-5) + 1e-5 / c.numel())
    u, v, g = logr.clone(), logc.clone(), 0.0
    t = min(16.0, gamma)
    while True:
        if g:  # potentials grow with gamma
            u, v = u * (t / g), v * (t / g)
        for _ in range(2 if t < gamma else 4):
            u = logr - _lse_rows(v, C, X, Y, t, scale)
            v = logc - _lse_rows(u, Ct, Y, X, t, scale)
        g = t
        if t >= gamma:
            return u.contiguous(), v.contiguous()
        t = min(gamma, 4.0 * t)


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        rng = np.random.Generator(np.random.PCG64(case["count"] * 7919 + case["lo"]))
        sizes = rng.integers(case["lo"], case["hi"] + 1, size=case["count"])  # the sizes belong to the case
        probs = []
        for k, n in enumerate(sizes):
            _, X, Y, r, c, _ = _make(dict(case, n=int(n), m=int(n)), seed * 1009 + k)
            probs.append(E.Problem(X=X, Y=Y, r=r, c=c, precision="mixed"))
        h = E.Handle(0, int(sizes.max()), int(sizes.max()), case["d"])
        return dict(case=case, h=h, probs=probs, params=_params(case))
    C, X, Y, r, c, scale = _make(case, seed)
    n, m = case["n"], case["m"]
    h = E.Handle(0, n, m, case.get("d", 0))
    s = dict(case=case, h=h, r=r, c=c)
    if op in ("solve", "train"):
        s["params"] = _params(case)
        if op == "solve":
            s["prob"] = E.Problem(C=C, X=X, Y=Y, r=r, c=c, precision=case["prec"])
        else:
            s["C"], s["X"], s["Y"] = (t if t is None else t.requires_grad_() for t in (C, X, Y))
        return s
    s["u"], s["v"] = _potentials(C, X, Y, r, c, case["gamma"], scale)
    s["prob"] = E.Problem(C=C, X=X, Y=Y, r=r, c=c, precision=case["prec"], cost_scale=scale)
    if op == "hvp":
        gen = torch.Generator(device=DEV).manual_seed(int(seed) + 5)
        s["du"] = torch.randn(n, generator=gen, dtype=F64, device=DEV)
        s["dv"] = torch.randn(m, generator=gen, dtype=F64, device=DEV)
    return s


def _params(case):
    return E.default_params(gamma_i=16.0, gamma_f=case["gamma"], tol_final=1e-6)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case, h = state["case"], state["h"]
    op, gamma = case["op"], case["gamma"]
    if op == "marginals":
        return h.marginals(state["prob"], state["u"], state["v"], gamma)
    if op == "hvp":
        return h.hvp(state["prob"], state["u"], state["v"], gamma, 0.9, state["du"], state["dv"])
    if op == "backward":
        prob, u, v = state["prob"], state["u"], state["v"]
        if prob.C is not None:
            dC = torch.empty(prob.n, prob.m, device=DEV)
            dr, dc = torch.empty_like(u), torch.empty_like(v)
            h.eot_backward(prob, u, v, gamma, dC=dC, dr=dr, dc=dc)
            return dC, dr, dc
        dX, dY = torch.empty(prob.n, prob.d, device=DEV), torch.empty(prob.m, prob.d, device=DEV)
        dr, dc = torch.empty_like(u), torch.empty_like(v)
        h.eot_backward(prob, u, v, gamma, dX=dX, dY=dY, dr=dr, dc=dc)
        return dX, dY, dr, dc
    if op == "match":
        prob, u, v = state["prob"], state["u"], state["v"]
        best = torch.empty(prob.n, dtype=torch.int64, device=DEV)
        rows = torch.empty(prob.n, dtype=torch.int64, device=DEV)
        total = torch.empty(1, dtype=torch.int64, device=DEV)
        h.eot_plan_argmax(prob, v, gamma, best)
        # the entries above a hundredth of the uniform plan's
        h.eot_plan_support(prob, u, v, gamma, math.log(0.01 / (prob.n * prob.m)), rows, total)
        return best, rows, total
    if op == "round":
        prob, u, v = state["prob"], state["u"], state["v"]
        u1, v1, a, b = torch.empty_like(u), torch.empty_like(v), torch.empty_like(u), torch.empty_like(v)
        cost, corr = h.eot_round(prob, u, v, gamma, u1, v1, a, b)
        return cost, corr, u1, v1, a, b
    if op == "solve":
        u, v, _ = h.solve(state["prob"], state["params"])
        value = torch.empty((), dtype=F64, device=DEV)
        h.eot_value(state["prob"], u, v, gamma, value)
        return value, u, v
    if op == "train":
        C, X, Y = state["C"], state["X"], state["Y"]
        value, _, _ = E.eot_value(h, state["r"], state["c"], C=C, X=X, Y=Y, precision=case["prec"],
                                  params=state["params"])
        leaves = (C,) if C is not None else (X, Y)
        loss = value.to(leaves[0].dtype)  # joins the loss of the float32 model that makes the leaves
        return (loss.detach(),) + torch.autograd.grad(loss, leaves)
    probs = state["probs"]
    us, vs, status, _ = E.solve_batched(h, probs, state["params"])
    n, m, d = sum(p.n for p in probs), sum(p.m for p in probs), case["d"]
    dX, dY = torch.empty(n, d, device=DEV), torch.empty(m, d, device=DEV)
    values = torch.empty(len(probs), dtype=F64, device=DEV)
    i = j = 0
    for k, p in enumerate(probs):
        h.eot_value(p, us[k], vs[k], gamma, values[k])
        h.eot_backward(p, us[k], vs[k], gamma, dX=dX[i:i + p.n], dY=dY[j:j + p.m])
        i, j = i + p.n, j + p.m
    return values.float(), dX, dY, torch.tensor(status)


# ---------------------------------------------------------------------------
# what a pass cannot do without, and its outputs in 64 bits
# ---------------------------------------------------------------------------

def work(case):
    """Each input read once, each output written once; operations of the sweeps that one
    call needs (a solve: of one row and one column sweep, however many it takes)."""
    op = case["op"]
    if op == "batch":
        mean = (case["lo"] + case["hi"]) / 2.0
        entries, sides, d = case["count"] * mean * mean, case["count"] * 2.0 * mean, case["d"]
        return {"bytes": sides * (4.0 * d + 8.0 + 4.0 * d), "flops": entries * 4.0 * (3.0 * d + 6.0)}
    n, m, d = case["n"], case["m"], case.get("d", 0)
    size = 8.0 if case["prec"] == "fp64" else 4.0
    form = 3.0 * d + 4.0 if d else 4.0  # the exponent and its exponential
    data = 4.0 * d * (n + m) if d else size * n * m
    vec = 8.0 * (n + m)
    if op == "marginals":
        return {"bytes": data + 3 * vec, "flops": n * m * (form + 2.0)}
    if op == "hvp":
        return {"bytes": data + 4 * vec, "flops": n * m * (form + 8.0)}
    if op == "backward":
        out = 4.0 * d * (n + m) if d else 4.0 * n * m
        return {"bytes": data + out + 2 * vec, "flops": n * m * (form + 4.0 * d)}
    if op == "match":
        return {"bytes": data + 3 * vec, "flops": n * m * (form + 2.0)}
    if op == "round":
        return {"bytes": data + 4 * vec, "flops": 3.0 * n * m * (form + 4.0)}
    out = 0.0
    if op == "train":
        out = 4.0 * d * (n + m) if d else 4.0 * n * m
    return {"bytes": data + out + 2 * vec, "flops": 2.0 * n * m * (form + 2.0)}


def _blocks(C, X, Y, scale):
    """(first row, C of a block of rows) in 64 bits."""
    n, m = (C.shape if C is not None else (X.shape[0], Y.shape[0]))
    step = max(1, (1 << 25) // m)
    for i in range(0, n, step):
        if C is not None:
            yield i, C[i:i + step].double()
        else:
            D = torch.zeros(min(step, n - i), m, dtype=F64, device=DEV)
            for k in range(X.shape[1]):
                D += (X[i:i + step, k, None].double() - Y[None, :, k].double()) ** 2
            yield i, D.mul_(scale)


def _newton_value(C, r, c, gamma):
    """F* = <P*, C> - H(P*) / gamma of a small dense problem, to machine precision: dense
    Newton steps on the dual along a rising gamma, each after a few Sinkhorn steps."""
    keep_r, keep_c = r > 0, c > 0
    C, r, c = C.double()[keep_r][:, keep_c], r[keep_r], c[keep_c]
    logr, logc = torch.log(r), torch.log(c)
    u, v, g, t = logr.clone(), logc.clone(), 0.0, min(16.0, gamma)
    while True:
        if g:
            u, v = u * (t / g), v * (t / g)
        for step in range(60):
            for _ in range(4):
                u = logr - torch.logsumexp(v[None, :] - t * C, 1)
                v = logc - torch.logsumexp(u[:, None] - t * C, 0)
            P = torch.exp(u[:, None] + v[None, :] - t * C)
            rp = P.sum(1)
            err = float((rp - r).abs().sum())
            if err < (1e-6 if t < gamma else 1e-13):
                break
            S = torch.diag(rp) - (P / c[None, :]) @ P.T + rp[:, None] * rp[None, :]
            du = torch.linalg.solve(S, r - rp)
            u = u + du * min(1.0, 2.0 / float(du.abs().max()))
        v = logc - torch.logsumexp(u[:, None] - t * C, 0)
        if t >= gamma:
            return (r @ u + c @ v) / t  # the plan's mass is 1 after the column step
        g, t = t, min(gamma, 2.0 * t)


def exact(case, seed):
    op, gamma = case["op"], case["gamma"]
    if op in ("batch", "match"):
        return None  # whole numbers, or solves of many problems
    C, X, Y, r, c, scale = _make(case, seed)
    n, m = case["n"], case["m"]
    if op in ("solve", "train"):
        # a solve stops at a tolerance: its value has a limit to be held to (it is
        # stationary there), the potentials and gradients of its last iterate have not
        if n * m > 1100 * 1100:
            return None
        if C is None:
            D = torch.cat([b for _, b in _blocks(None, X, Y, 1.0)])
            C = D / D.max()
        return [_newton_value(C, r, c, gamma), None, None]
    u, v = _potentials(C, X, Y, r, c, gamma, scale)
    rp, cp = torch.zeros(n, dtype=F64, device=DEV), torch.zeros(m, dtype=F64, device=DEV)
    if op in ("marginals", "hvp"):
        if op == "hvp":
            gen = torch.Generator(device=DEV).manual_seed(int(seed) + 5)
            du = torch.randn(n, generator=gen, dtype=F64, device=DEV)
            dv = torch.randn(m, generator=gen, dtype=F64, device=DEV)
            pdv, ptdu = torch.zeros_like(rp), torch.zeros_like(cp)
        for i, B in _blocks(C, X, Y, scale):
            e = i + B.shape[0]
            P = torch.exp(u[i:e, None] + v[None, :] - gamma * B)
            rp[i:e] = P.sum(1)
            cp += P.sum(0)
            if op == "hvp":
                pdv[i:e] = P @ dv
                ptdu += P.T @ du[i:e]
        if op == "hvp":
            return [rp * du + 0.9 * pdv, 0.9 * ptdu + cp * dv, rp, cp]
        return [rp, cp, torch.log(rp), torch.log(cp), rp.sum().reshape(1)]
    if op == "backward":
        if C is not None:
            P = torch.exp(u[:, None] + v[None, :] - gamma * C.double())
            return [P, u / gamma, v / gamma]
        X64, Y64 = X.double(), Y.double()
        dX, dY = torch.zeros_like(X64), torch.zeros_like(Y64)
        for i, B in _blocks(C, X, Y, scale):
            e = i + B.shape[0]
            P = torch.exp(u[i:e, None] + v[None, :] - gamma * B)
            for k in range(X.shape[1]):
                G = P * (X64[i:e, k, None] - Y64[None, :, k])
                dX[i:e, k] = G.sum(1)
                dY[:, k] -= G.sum(0)
        return [2 * scale * dX, 2 * scale * dY, u / gamma, v / gamma]
    # round: scale rows then columns below their marginals, correct by a rank-one term
    for i, B in _blocks(C, X, Y, scale):
        e = i + B.shape[0]
        rp[i:e] = torch.exp(u[i:e, None] + v[None, :] - gamma * B).sum(1)
    x = torch.where(rp <= r, torch.ones_like(r), r / rp)
    for i, B in _blocks(C, X, Y, scale):
        e = i + B.shape[0]
        cp += x[i:e] @ torch.exp(u[i:e, None] + v[None, :] - gamma * B)
    y = torch.where(cp <= c, torch.ones_like(c), c / cp)
    b = c - y * cp
    a, cost, cb = torch.zeros_like(r), 0.0, torch.zeros_like(r)
    for i, B in _blocks(C, X, Y, scale):
        e = i + B.shape[0]
        F = x[i:e, None] * torch.exp(u[i:e, None] + v[None, :] - gamma * B) * y[None, :]
        a[i:e] = r[i:e] - F.sum(1)
        cost += float((B * F).sum())
        cb[i:e] = B @ b
    corr = float(a.abs().sum())
    return [cost + float(a @ cb) / corr, corr, u + torch.log(x), v + torch.log(y), a, b]
