"""Accuracy of the tensor-core point sweeps (17 <= d <= 64) over the temperatures that the
library accepts, and where the digits' extra bits are not available."""
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


def balanced(C, gamma):
    """Potentials of a plan: Sinkhorn steps along a rising gamma, columns last."""
    n, m = C.shape
    u, v, g = np.zeros(n), np.zeros(m), 16.0
    while True:
        for _ in range(20):
            u = -np.log(n) - O.lse_r(v[None, :] - g * C)
            v = -np.log(m) - O.lse_c(u[:, None] - g * C)
        if g >= gamma:
            return u, v
        g, f = min(2.0 * g, gamma), min(2.0, gamma / g)
        u, v = u * f, v * f


@pytest.mark.parametrize("e", [8, 10, 12, 14, 16, 18])
@pytest.mark.parametrize("kind,d,shift", [("uniform", 17, 0.0), ("uniform", 64, 0.0), ("gaussians", 33, 0.0),
                                          ("gaussians", 64, 0.0), ("uniform", 20, 5.0), ("gaussians", 64, 20.0),
                                          ("corners", 64, 0.0), ("corners", 32, 0.0)])
def test_marginals_and_products(H, e, kind, d, shift, monkeypatch):
    """The two LSE sweeps and the two weighted sweeps (Hessian-vector product) against 64
    bits. L1 errors relative to the sum of absolute terms: at most 1.5 times the general
    sweeps' (EOT_TC=0: FP32 exponents and exponentials as here) plus 2e-8, a sixth of an
    FP32 rounding, plus twice the digits' rounding of the coordinates, 1.2e-7 at gamma =
    2^18 (four times that without extra bits: clouds on the corners of a cube, the case
    in which the level sums reach 2^24)."""
    from paper_2504_02067_gb300 import Problem
    n, m = 300, 260
    rng = np.random.default_rng(d + e)
    if kind == "uniform":
        X, Y = (rng.uniform(0, 1, size=(k, d)) for k in (n, m))
    elif kind == "gaussians":
        mu = 2.0 * rng.normal(size=(8, d))
        X, Y = (mu[rng.integers(0, 8, size=k)] + rng.normal(size=(k, d)) for k in (n, m))
    else:  # corners, each moved by up to a part in 50; the first (the common centre) in the middle
        sg = rng.choice([-1.0, 1.0], size=(12, d))
        X, Y = (sg[rng.integers(0, 12, size=k)] * (1.0 - 0.02 * rng.uniform(0, 1, size=(k, d))) for k in (n, m))
        X[0] = 0.0
        X[1], Y[1] = 0.9999, -0.9999
    Y[:, 0] += shift
    X, Y = X.astype(np.float32), Y.astype(np.float32)
    gamma = 2.0 ** e
    sC = O.sqeuclid_scale(X, Y)
    C = sC * O.sqeuclid(X, Y)
    u, v = balanced(C, gamma)
    P = np.exp(u[:, None] + v[None, :] - gamma * C)
    du, dv = rng.normal(size=n), rng.normal(size=m)
    prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), precision="mixed", cost_scale=sC)
    r, c = P.sum(1), P.sum(0)
    def run(flag):
        monkeypatch.setenv("EOT_TC", flag)
        mg = H.marginals(prob, t(u), t(v), gamma)
        hv = H.hvp(prob, t(u), t(v), gamma, 0.9, t(du), t(dv))
        return [x.cpu().numpy() for x in (mg[0], mg[1], hv[0], hv[1])]

    want = [r, c, r * du + 0.9 * (P @ dv), 0.9 * (P.T @ du) + c * dv]
    size = [r, c, np.abs(r * du) + 0.9 * (P @ np.abs(dv)), 0.9 * (P.T @ np.abs(du)) + np.abs(c * dv)]
    digits = (4.8e-7 if kind == "corners" else 1.2e-7) * gamma / 2.0 ** 18
    for k, (a, b, w, z) in enumerate(zip(run("1"), run("0"), want, size)):
        ea, eb = np.abs(a - w).sum() / z.sum(), np.abs(b - w).sum() / z.sum()
        print("%s %d 2^%d [%d] %.2e general %.2e" % (kind, d, e, k, ea, eb))
        assert ea <= 1.5 * eb + 2e-8 + digits, (k, ea, eb, digits)
