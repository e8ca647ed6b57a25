"""The point-cost maximum at the edges of its blocks and tiles."""
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


@pytest.mark.parametrize("n,m,d", [(1, 2, 1), (127, 63, 64), (129, 65, 33), (128, 64, 17), (300, 257, 16), (513, 1025, 4),
                                   (2000, 130, 5)])
@pytest.mark.parametrize("where", ["first", "last", "middle"])
def test_cost_scale_is_the_farthest_pair(H, n, m, d, where):
    """The library's own normalisation against the same call with 1 / max_ij |x_i - y_j|^2
    given: the farthest pair is found wherever it lies (its cost to FP64 rounding, an
    exponent below 64, so 1e-12)."""
    from paper_2504_02067_gb300 import Problem
    rng = np.random.default_rng(n + m + d)
    X, Y = (rng.uniform(0, 1, size=(k, d)).astype(np.float32) for k in (n, m))
    i, j = {"first": (0, 0), "last": (n - 1, m - 1), "middle": (n // 2, m // 2)}[where]
    X[i] += 3.0
    Y[j] -= 2.0
    sC = O.sqeuclid_scale(X, Y)
    one = [Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), r=t(np.full(n, 1.0 / n)), c=t(np.full(m, 1.0 / m)),
                   precision="fp64", cost_scale=s) for s in (0.0, sC)]
    a, b = [[x.cpu().numpy() for x in H.marginals(p, t(np.zeros(n)), t(np.zeros(m)), 64.0)[:2]] for p in one]
    for x, y in zip(a, b):
        assert (np.abs(x - y) <= 1e-12 * np.abs(y)).all()
