"""The screened integer outputs (argmax, support) at the ends of the screening's reach.
Whole numbers, so every comparison with the oracle is exact."""
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


def argmax(H, prob, v, gamma):
    idx = torch.full((prob.n,), -7, dtype=torch.int64, device=DEV)
    H.eot_plan_argmax(prob, t(v), gamma, idx)
    return idx.cpu().numpy()


@pytest.mark.parametrize("f64", [False, True])
def test_dense_maximum_that_comes_into_reach_late(H, f64):
    """Row maxima around -1e8: the screening passes over entries below it, and a later
    entry whose FP32 value is just above it must not hide one of them that is larger."""
    from paper_2504_02067_gb300 import Problem
    n, m = 64, 4096
    C = np.full((n, m), 3.0e8)
    v = np.zeros(m)
    C[:, 0] = 100000008.0 - 8.0 * (np.arange(n) - n // 2)
    v[1000] = -67108871.0
    C[:, 1000] = 32891141.9 - 8.0 * (np.arange(n) - n // 2)
    C = C if f64 else C.astype(np.float32)
    prob = Problem(t(C, torch.float64 if f64 else torch.float32), precision="fp64" if f64 else "mixed")
    assert np.array_equal(argmax(H, prob, v, 1.0), O.plan_row_argmax(v, 1.0, C.astype(np.float64)))


def test_point_maximum_that_comes_into_reach_late(H):
    """The same through the point kernel, the two contenders in different tiles of a
    cluster's chunks and of one chunk."""
    from paper_2504_02067_gb300 import Problem
    X = np.zeros((70, 3), dtype=np.float32)
    for m in (1500, 200000):
        Y = np.zeros((m, 3), dtype=np.float32)
        Y[:, 2] = 20000.0
        Y[0] = 2.0, 1.0, 10000.0  # exponent -100000005, in FP32 -100000008
        Y[1000, 2] = 5735.0       # exponent -100000008.9, in FP32 -100000000
        v = np.full(m, -np.inf)   # (the other columns have no mass)
        v[0], v[1000] = 0.0, -67109783.9
        prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), precision="mixed", cost_scale=1.0)
        C = np.concatenate([O.sqeuclid_ordered(X, Y[k:k + 10000]) for k in range(0, m, 10000)], axis=1)
        assert np.array_equal(argmax(H, prob, v, 1.0), O.plan_row_argmax(v, 1.0, C)), m


def support(H, prob, u, v, gamma, log_tau):
    cnt = torch.full((prob.n,), -7, dtype=torch.int64, device=DEV)
    tot = torch.full((1,), -7, dtype=torch.int64, device=DEV)
    H.eot_plan_support(prob, t(u), t(v), gamma, log_tau, cnt, tot)
    cnt = cnt.cpu().numpy()
    assert int(tot.item()) == int(cnt.sum())
    return cnt


@pytest.mark.parametrize("m", [130, 4096, 4099])
def test_gamma_zero_with_costs_beyond_fp32(H, m):
    """gamma = 0: every exponent is v_j (argmax) or u_i + v_j (support), also where the
    cost overflows FP32 (a dense FP64 cost of 1e39, coordinates 1e20 apart)."""
    from paper_2504_02067_gb300 import Problem
    rng = np.random.default_rng(m)
    n = 70
    u, v = rng.normal(size=n), rng.normal(size=m)
    C = rng.uniform(0, 1, size=(n, m))
    C[:, ::3] = 1.0e39
    X, Y = rng.normal(size=(n, 2)).astype(np.float32), rng.normal(size=(m, 2)).astype(np.float32)
    Y[::3, 1] = 1.0e20
    for prob, cost in ((Problem(t(C), precision="fp64"), C),
                       (Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), precision="mixed", cost_scale=1.0),
                        O.sqeuclid_ordered(X, Y))):
        assert np.array_equal(argmax(H, prob, v, 0.0), O.plan_row_argmax(v, 0.0, cost))
        for log_tau in (-0.5, 0.0, 1.0):
            assert np.array_equal(support(H, prob, u, v, 0.0, log_tau), O.plan_support_counts(u, v, 0.0, cost, log_tau))


def test_potentials_beyond_fp32(H):
    """Finite potentials below FP32's range beside costs as large and negative."""
    from paper_2504_02067_gb300 import Problem
    rng = np.random.default_rng(4)
    n, m = 9, 700
    u, v, C = rng.normal(size=n), rng.normal(size=m), rng.uniform(0, 1, size=(n, m))
    v[5] = -1.0e39
    C[:, 5] = -1.0e38
    C[::2, 5] = -2.0e37
    prob = Problem(t(C), precision="fp64")
    assert np.array_equal(argmax(H, prob, v, 20.0), O.plan_row_argmax(v, 20.0, C))
    assert np.array_equal(support(H, prob, u, v, 20.0, -1.0), O.plan_support_counts(u, v, 20.0, C, -1.0))


def test_costs_below_fp32_at_a_large_gamma(H):
    """FP64 costs below 2^-126 whose product with gamma decides."""
    from paper_2504_02067_gb300 import Problem
    rng = np.random.default_rng(5)
    n, m, gamma = 33, 1001, 1.0e30
    C = rng.uniform(0, 1, size=(n, m)) * 2.0 ** -127
    u, v = np.zeros(n), rng.uniform(0, 1e-9, size=m)
    prob = Problem(t(C), precision="fp64")
    assert np.array_equal(argmax(H, prob, v, gamma), O.plan_row_argmax(v, gamma, C))
    for log_tau in (-5e-9, -2e-9, 0.0):
        assert np.array_equal(support(H, prob, u, v, gamma, log_tau), O.plan_support_counts(u, v, gamma, C, log_tau))


@pytest.mark.parametrize("n,m,d", [(1, 20, 2), (70, 129, 3), (130, 1100, 3), (65, 2050, 40)])
def test_points_with_many_repeats(H, n, m, d):
    """Clouds of few distinct points: every row has more ties and open entries than the
    screening keeps, in every chunk of the columns; some rows have no mass."""
    from paper_2504_02067_gb300 import Problem
    rng = np.random.default_rng(m + d)
    base = rng.integers(0, 4, size=(5, d))
    X, Y = (base[rng.integers(0, 5, size=k)].astype(np.float32) for k in (n, m))
    u, v = rng.normal(size=n), np.zeros(m)
    v[rng.choice(m, m // 3, replace=False)] = -np.inf
    u[rng.choice(n, n // 4, replace=False)] = -np.inf
    sC = O.sqeuclid_scale(X, Y) if n > 1 else 0.25
    prob = Problem(X=t(X, torch.float32), Y=t(Y, torch.float32), precision="mixed", cost_scale=sC)
    C = sC * O.sqeuclid_ordered(X, Y)
    for gamma in (0.0, 64.0):
        assert np.array_equal(argmax(H, prob, v, gamma), O.plan_row_argmax(v, gamma, C))
        on = float(u[np.isfinite(u)][0]) - gamma * float(C.min()) if np.isfinite(u).any() else -1.0
        for log_tau in (on, -1.0, -np.inf):
            with np.errstate(invalid="ignore"):
                want = O.plan_support_counts(u, v, gamma, C, log_tau)
            assert np.array_equal(support(H, prob, u, v, gamma, log_tau), want)
