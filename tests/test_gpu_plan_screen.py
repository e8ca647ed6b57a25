"""The screened integer outputs (argmax, support) where the screening can go wrong:
tile and chunk edges, rows full of near ties, masses of -inf, potentials beyond
the screening's range, temperatures beyond it, unaligned rows. Whole numbers, so
every comparison with the oracle is exact."""
import math

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


def check(H, prob, C64, u, v, gamma):
    with np.errstate(invalid="ignore"):
        t_all = (u[:, None] + v[None, :]) - gamma * C64
    fin = t_all[np.isfinite(t_all)]
    idx = torch.full((prob.n,), -7, dtype=torch.int64, device=DEV)
    H.eot_plan_argmax(prob, t(v), gamma, idx)
    assert np.array_equal(idx.cpu().numpy(), O.plan_row_argmax(v, gamma, C64))
    # thresholds in the bulk, on an entry, above and below everything
    for log_tau in (float(np.quantile(fin, 0.6)), float(fin[fin.size // 2]), float(fin.max()) + 1.0,
                    float(fin.min()) - 1.0, -math.inf):
        cnt = torch.full((prob.n,), -7, dtype=torch.int64, device=DEV)
        tot = torch.full((1,), -7, dtype=torch.int64, device=DEV)
        H.eot_plan_support(prob, t(u), t(v), gamma, log_tau, cnt, tot)
        ref = O.plan_support_counts(u, v, gamma, C64, log_tau)
        assert np.array_equal(cnt.cpu().numpy(), ref) and int(tot.item()) == int(ref.sum())


def potentials(rng, n, m, kind):
    u, v = rng.normal(0, 2, n), rng.normal(0, 2, m)
    if kind == "empty":  # columns and rows without mass
        v[rng.choice(m, m // 3, replace=False)] = -np.inf
        u[rng.choice(n, n // 5, replace=False)] = -np.inf
    if kind == "gauge":
        u, v = u - 3.0e5, v + 3.0e5
    if kind == "huge":  # beyond the screening: decided in FP64 throughout
        v[m // 2] = 1.0e12
        u[0] = -2.0e9
    if kind == "flat":
        u[:], v[:] = 0.0, 0.0
    return u, v


@pytest.mark.parametrize("n,m", [(1, 4097), (9, 513), (64, 4100), (65, 129), (130, 8200)])
@pytest.mark.parametrize("kind", ["plain", "empty", "gauge", "huge", "flat"])
@pytest.mark.parametrize("f64", [False, True])
def test_dense_screen(H, n, m, kind, f64):
    from paper_2504_02067_gb300 import Problem
    rng = np.random.default_rng(n * 7 + m)
    C = rng.integers(0, 12, size=(n, m)) / 11.0 if kind == "flat" else rng.uniform(0, 1, size=(n, m))
    C = C if f64 else C.astype(np.float32)
    u, v = potentials(rng, n, m, kind)
    prob = Problem(t(C, torch.float64 if f64 else torch.float32), precision="fp64" if f64 else "mixed")
    check(H, prob, C.astype(np.float64), u, v, 300.0)
    if kind == "plain":
        for gamma in (0.0, 1e-40, 1e-3):
            check(H, prob, C.astype(np.float64), u, v, gamma)
        # rows that are not 16-byte aligned
        wide = torch.zeros(n, m + 3, dtype=prob.C.dtype, device=DEV)
        wide[:, 1:m + 1] = prob.C
        check(H, Problem(wide[:, 1:m + 1], precision=prob.precision), C.astype(np.float64), u, v, 300.0)


@pytest.mark.parametrize("n,m,d", [(1, 129, 1), (65, 1000, 2), (64, 128, 31), (63, 2050, 33), (200, 300, 64),
                                   (700, 1025, 5)])
@pytest.mark.parametrize("kind", ["plain", "empty", "gauge", "huge", "flat"])
def test_point_screen(H, n, m, d, kind):
    from paper_2504_02067_gb300 import Problem
    rng = np.random.default_rng(n + 7 * m + d)
    if kind == "flat":  # lattice points with equal potentials: many exact ties per row
        X, Y = rng.integers(0, 3, size=(n, d)), rng.integers(0, 3, size=(m, d))
    else:
        X, Y = rng.normal(0, 1, size=(n, d)) + 5.0, rng.normal(0, 1, size=(m, d)) + 5.2
    X, Y = X.astype(np.float32), Y.astype(np.float32)
    u, v = potentials(rng, n, m, kind)
    sC = O.sqeuclid_scale(X, Y)
    prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), precision="mixed", cost_scale=sC)
    C64 = sC * O.sqeuclid_ordered(X, Y)
    check(H, prob, C64, u, v, 300.0)
    if kind == "plain":
        check(H, prob, C64, u, v, 0.0)
