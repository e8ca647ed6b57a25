"""The split-coordinate point sweeps (csrc/sweep_pgrid.cuh) against the general point
sweeps and the oracle, at the sizes where the work split changes (one warp of own
elements, warp groups, clusters, one thread owning four) and in every dimension
class, with clouds off the origin and gauge-shifted potentials."""
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


SIZES = [(1, 1, 1), (5, 300, 2), (33, 31, 3), (700, 1000, 2), (257, 2050, 4), (130, 90, 5), (300, 517, 8),
         (1100, 900, 9), (400, 333, 16), (6000, 5000, 3)]


@pytest.mark.parametrize("n,m,d", SIZES)
@pytest.mark.parametrize("offset,gauge", [(0.0, 0.0), (1000.0, 0.0), (3.0, 2.0e5)])
@pytest.mark.parametrize("given", [False, True])
def test_sweeps_against_oracle_and_general(H, n, m, d, offset, gauge, given):
    """Marginals (the two LSE sweeps), HVP (two weighted sweeps) and gradients. Bounds:
    marginals L1 1e-6 (the library's bound for the mixed path); HVP and gradients
    within 1e-5 of the sum of absolute terms; and the error against the oracle at
    most 1.5 times the general sweeps' plus 1e-7 (FP32 rounding of either)."""
    from paper_2504_02067_gb300 import Problem
    rng = np.random.default_rng(n + 3 * m + d)
    X = (rng.uniform(0, 1, size=(n, d)) + offset).astype(np.float32)
    Y = (rng.uniform(0, 1, size=(m, d)) + offset).astype(np.float32)
    if n == 1 and m == 1:
        Y = X + np.float32(0.5)
    gamma = 512.0
    sC = O.sqeuclid_scale(X, Y)
    C = sC * O.sqeuclid(X, Y)
    u = rng.normal(0, 0.5, n)
    # potentials of a plan: the columns sum to about 1 / m
    M = u[:, None] - gamma * C
    v = -np.log(m) - (M.max(0) + np.log(np.exp(M - M.max(0)).sum(0)))
    P = np.exp(u[:, None] + v[None, :] - gamma * C)
    u, v = u + gauge, v - gauge
    r, c = P.sum(1), P.sum(0)
    prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), r=t(r / r.sum()), c=t(c / c.sum()),
                   precision="mixed", cost_scale=sC if given else 0.0)
    du, dv = rng.normal(size=n), rng.normal(size=m)

    def run():
        mg = H.marginals(prob, t(u), t(v), gamma)
        hv = H.hvp(prob, t(u), t(v), gamma, 0.9, t(du), t(dv))
        dX, dY = (torch.empty(k, d, dtype=torch.float32, device=DEV) for k in (n, m))
        H.eot_backward(prob, t(u), t(v), gamma, dX=dX, dY=dY)
        return [x.cpu().numpy() for x in (mg[0], mg[1], hv[0], hv[1], dX, dY)]

    D = X[:, None, :].astype(np.float64) - Y[None, :, :]
    want = [r, c, r * du + 0.9 * (P @ dv), 0.9 * (P.T @ du) + c * dv,
            2 * sC * np.einsum("ij,ijk->ik", P, D), -2 * sC * np.einsum("ij,ijk->jk", P, D)]
    size = [r, c, np.abs(r * du) + 0.9 * (P @ np.abs(dv)), 0.9 * (P.T @ np.abs(du)) + np.abs(c * dv),
            2 * sC * np.einsum("ij,ijk->ik", P, np.abs(D)), 2 * sC * np.einsum("ij,ijk->jk", P, np.abs(D))]
    got, gen = run(), general(run)
    for k, (a, b, w, z) in enumerate(zip(got, gen, want, size)):
        ea, eb = np.abs(a - w).sum() / z.sum(), np.abs(b - w).sum() / z.sum()
        assert ea <= (1e-6 if k < 2 else 1e-5), (k, ea, eb)
        assert ea <= 1.5 * eb + 1e-7, (k, ea, eb)
        assert (np.abs(a - w) <= 1e-5 * z + 1e-30).all(), k


@pytest.mark.parametrize("n,m,d", [(300, 260, 2), (900, 1100, 3), (150, 400, 9)])
def test_solve_reaches_tolerance(H, n, m, d):
    """A full solve ends at marginal L1 <= 1e-6 as the oracle measures it, with the
    general sweeps' stage count (the schedule does not see rounding)."""
    from paper_2504_02067_gb300 import Problem, default_params
    rng = np.random.default_rng(5 * n + d)
    X, Y = (rng.uniform(0, 1, size=(k, d)).astype(np.float32) for k in (n, m))
    r, c = rng.dirichlet(np.ones(n)), rng.dirichlet(np.ones(m))
    prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), r=t(r), c=t(c), precision="mixed")
    prm = default_params(gamma_i=16.0, gamma_f=1024.0)
    u, v, st = H.solve(prob, prm)
    _, _, sg = general(lambda: H.solve(prob, prm))
    assert st["stages"] == sg["stages"]
    C = O.sqeuclid_scale(X, Y) * O.sqeuclid(X, Y)
    assert O.marginal_l1_error(u.cpu().numpy(), v.cpu().numpy(), 1024.0, C, r, c) <= 1e-6


def test_beyond_the_bound_takes_the_general_sweeps(H):
    """A scale that puts gamma s_C max |x - y|^2 beyond the split's range gives the
    general sweeps' bits."""
    from paper_2504_02067_gb300 import Problem
    rng = np.random.default_rng(3)
    X, Y = (rng.uniform(0, 1, size=(k, 2)).astype(np.float32) for k in (90, 70))
    prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), precision="mixed", cost_scale=400.0)
    u, v = t(rng.normal(size=90)), t(rng.normal(size=70))
    a = H.marginals(prob, u, v, 512.0)
    b = general(lambda: H.marginals(prob, u, v, 512.0))
    assert all(torch.equal(x, y) for x, y in zip(a, b))
