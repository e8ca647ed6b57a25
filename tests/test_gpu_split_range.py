"""The split-coordinate point sweeps (csrc/sweep_pgrid.cuh) at the ends of their range:
temperatures too small for their scaled coordinates, coinciding points, and solves
whose stages cross from them to the general sweeps."""
import os

import numpy as np
import pytest

from oracle import eot_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_02067_gb300 import Handle, build
    build()
    h = Handle(0, 64, 64)
    yield h
    h.close()


def t(x, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x)).to(device=DEV, dtype=dtype)


def general(fn):
    """fn on the general point sweeps."""
    os.environ["EOT_PGRID"] = "0"
    try:
        return fn()
    finally:
        del os.environ["EOT_PGRID"]


@pytest.mark.parametrize("d", [2, 9, 33])
@pytest.mark.parametrize("gamma", [1e-50, 1e-30, 1e-12])
def test_gradients_at_a_tiny_gamma(H, d, gamma):
    """P = exp(u + v) there: each component within 1e-5 of the sum of absolute terms
    (the bound of the mixed gradients)."""
    from paper_2504_02067_gb300 import Problem
    n, m = 60, 45
    rng = np.random.default_rng(d)
    X, Y = (rng.normal(size=(k, d)).astype(np.float32) for k in (n, m))
    u, v = np.log(rng.dirichlet(np.ones(n))), np.log(rng.dirichlet(np.ones(m)))
    P = np.exp(u[:, None] + v[None, :])
    D = X[:, None, :].astype(np.float64) - Y[None].astype(np.float64)
    for sC in (0.0, 0.5):
        s = sC or O.sqeuclid_scale(X, Y)
        prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), precision="mixed", cost_scale=sC)
        dX, dY = (torch.empty(k, d, dtype=torch.float32, device=DEV) for k in (n, m))
        H.eot_backward(prob, t(u), t(v), gamma, dX=dX, dY=dY)
        for got, ax, sg in ((dX, 1, 1.0), (dY, 0, -1.0)):
            want = sg * 2 * s * (P[:, :, None] * D).sum(ax)
            size = 2 * s * (P[:, :, None] * np.abs(D)).sum(ax)
            assert (np.abs(got.cpu().numpy() - want) <= 1e-5 * size).all()


def test_batched_coinciding_points_with_a_given_scale(H):
    """A cost that is zero throughout: the product plan."""
    from paper_2504_02067_gb300 import Problem, default_params, solve_batched
    rng = np.random.default_rng(2)
    n, m = 40, 70
    r, c = rng.dirichlet(np.ones(n)), rng.dirichlet(np.ones(m))
    X, Y = np.full((n, 2), 0.3, dtype=np.float32), np.full((m, 2), 0.3, dtype=np.float32)
    prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), r=t(r), c=t(c), precision="mixed", cost_scale=1.0)
    us, vs, st, _ = solve_batched(H, [prob], default_params(gamma_i=16.0, gamma_f=256.0))
    assert st == [0]
    P = np.exp(us[0].cpu().numpy()[:, None] + vs[0].cpu().numpy()[None, :])
    assert np.abs(P - r[:, None] * c[None, :]).sum() <= 2e-6


@pytest.mark.parametrize("n,m,d", [(200, 260, 2), (150, 130, 7)])
@pytest.mark.parametrize("gamma_f", [4096.0, 65536.0])
def test_solve_across_the_range(H, n, m, d, gamma_f):
    """The stages of one solve take different sweeps; it ends at marginal L1 <= 1e-6 as
    the oracle measures it, with the general sweeps' stage count."""
    from paper_2504_02067_gb300 import Problem, default_params, solve_batched
    rng = np.random.default_rng(n + d)
    X, Y = (rng.uniform(0, 1, size=(k, d)).astype(np.float32) for k in (n, m))
    r, c = (0.9 * rng.dirichlet(np.ones(k)) + 0.1 / k for k in (n, m))
    prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), r=t(r), c=t(c), precision="mixed")
    prm = default_params(gamma_i=16.0, gamma_f=gamma_f)
    C = O.sqeuclid_scale(X, Y) * O.sqeuclid(X, Y)
    u, v, st = H.solve(prob, prm)
    _, _, sg = general(lambda: H.solve(prob, prm))
    assert st["stages"] == sg["stages"]
    assert O.marginal_l1_error(u.cpu().numpy(), v.cpu().numpy(), gamma_f, C, r, c) <= 1e-6
    if d <= 4:
        us, vs, status, _ = solve_batched(H, [prob, prob], prm)
        assert status == [0, 0]
        for a, b in zip(us, vs):
            assert O.marginal_l1_error(a.cpu().numpy(), b.cpu().numpy(), gamma_f, C, r, c) <= 1e-6


@pytest.mark.parametrize("d", [1, 2, 3, 8, 16, 17, 33, 64])
@pytest.mark.parametrize("shift", [0.0, 5.0])
@pytest.mark.parametrize("gamma", [1400.0, 2600.0, 16384.0, 22000.0])
@pytest.mark.parametrize("given", [False, True])
def test_accuracy_over_the_range(H, d, shift, gamma, given):
    """Overlapping clouds, and one of them moved away so that every pair is far apart and
    the potentials cancel most of the cost. Errors against 64 bits, relative to the sum of
    absolute terms: at most 1.5 times the general sweeps' plus 2e-8, a sixth of an FP32
    rounding (the entries' own errors are smaller than the general sweeps'; in sums over
    entries the two schemes' roundings average differently)."""
    from paper_2504_02067_gb300 import Problem
    n, m = 300, 260
    rng = np.random.default_rng(d)
    X, Y = (rng.uniform(0, 1, size=(k, d)).astype(np.float32) for k in (n, m))
    Y[:, 0] += np.float32(shift)
    sC = O.sqeuclid_scale(X, Y)
    C = sC * O.sqeuclid(X, Y)
    u, v, g = np.zeros(n), np.zeros(m), 16.0
    while True:  # Sinkhorn steps along a rising gamma
        for _ in range(30):
            u = -np.log(n) - O.lse_r(v[None, :] - g * C)
            v = -np.log(m) - O.lse_c(u[:, None] - g * C)
        if g >= gamma:
            break
        g, f = min(2.0 * g, gamma), min(2.0, gamma / g)
        u, v = u * f, v * f
    P = np.exp(u[:, None] + v[None, :] - gamma * C)
    prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), precision="mixed", cost_scale=sC if given else 0.0)
    du, dv = rng.normal(size=n), rng.normal(size=m)

    def run():
        mg = H.marginals(prob, t(u), t(v), gamma)
        hv = H.hvp(prob, t(u), t(v), gamma, 0.9, t(du), t(dv))
        dX, dY = (torch.empty(k, d, dtype=torch.float32, device=DEV) for k in (n, m))
        H.eot_backward(prob, t(u), t(v), gamma, dX=dX, dY=dY)
        return [x.cpu().numpy() for x in (mg[0], mg[1], hv[0], hv[1], dX, dY)]

    D = X[:, None, :].astype(np.float64) - Y[None, :, :]
    r, c = P.sum(1), P.sum(0)
    want = [r, c, r * du + 0.9 * (P @ dv), 0.9 * (P.T @ du) + c * dv,
            2 * sC * np.einsum("ij,ijk->ik", P, D), -2 * sC * np.einsum("ij,ijk->jk", P, D)]
    size = [r, c, np.abs(r * du) + 0.9 * (P @ np.abs(dv)), 0.9 * (P.T @ np.abs(du)) + np.abs(c * dv),
            2 * sC * np.einsum("ij,ijk->ik", P, np.abs(D)), 2 * sC * np.einsum("ij,ijk->jk", P, np.abs(D))]
    got, gen = run(), general(run)
    for k, (a, b, w, z) in enumerate(zip(got, gen, want, size)):
        ea, eb = np.abs(a - w).sum() / z.sum(), np.abs(b - w).sum() / z.sum()
        assert ea <= 1.5 * eb + 2e-8, (k, ea, eb)
