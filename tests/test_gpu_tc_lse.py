"""The tensor-core LSE sweeps where their running maximum moves: within a tile, with
every tile, and not at all after the first, at tile and block edges."""
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


@pytest.mark.parametrize("n,m,d", [(128, 96, 17), (129, 97, 33), (500, 1111, 64), (1111, 500, 20)])
@pytest.mark.parametrize("order", ["far first", "near first", "mixed"])
def test_lse_where_the_maximum_moves(H, n, m, d, order):
    """Both clouds are sorted by distance from a corner, so the exponents rise (or fall,
    or jump) by hundreds of units along each sweep. The marginals are within the mixed
    path's bound: L1 error 1e-6 of the mass, and each of them within 4e-6 of itself
    (an exponent's FP32 rounding at its size below 32 and the FP32 sums)."""
    from paper_2504_02067_gb300 import Problem
    rng = np.random.default_rng(n + m + d)
    X = rng.uniform(0, 1, size=(n, d)).astype(np.float32)
    Y = rng.uniform(0, 1, size=(m, d)).astype(np.float32)
    for Z in (X, Y):
        k = np.argsort(-(Z.astype(np.float64) ** 2).sum(1))
        if order == "near first":
            k = k[::-1]
        elif order == "mixed":
            k = rng.permutation(len(k))
        Z[:] = Z[k]
    C = ((X[:, None, :].astype(np.float64) - Y[None].astype(np.float64)) ** 2).sum(-1)
    gamma = 64.0
    # v falls off from the corner too: exponents of one row span several hundred units
    v = -400.0 * (Y.astype(np.float64) ** 2).sum(1) / d
    u = np.log(1.0 / n) - O.lse_r(v[None, :] - gamma * C)
    P = np.exp(u[:, None] + v[None, :] - gamma * C)
    prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), cost_scale=1.0, r=t(np.full(n, 1.0 / n)),
                   c=t(np.full(m, 1.0 / m)), precision="mixed")
    r, c = [np.asarray(x.cpu()) for x in H.marginals(prob, t(u), t(v), gamma)[:2]]
    assert np.abs(r - P.sum(1)).sum() <= 1e-6
    assert np.abs(c - P.sum(0)).sum() <= 1e-6
    assert (np.abs(r - P.sum(1)) <= 4e-6 * P.sum(1)).all()
    assert (np.abs(c - P.sum(0)) <= 4e-6 * P.sum(0) + 1e-30).all()
