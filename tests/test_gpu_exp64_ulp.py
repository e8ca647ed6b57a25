"""The rounding of the FP64 sweeps' exponential (csrc/exp64.cuh), read off Round's row sums
as tests/test_gpu_exp64.py does, against the extended-precision exp of the host."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("lo,hi", [(-1.0, 1.0), (-8.0, 0.0), (-40.0, -8.0), (-300.0, -40.0), (-708.0, -300.0), (40.0, 600.0)])
def test_errors_are_those_of_a_rounding(lo, hi):
    """At most 0.9 ulp from the exact value (0.5 of it the result's own rounding; CUDA's exp
    reaches 0.87) and without a bias: a mean error below 0.02 ulp (a rounding's spread,
    0.29 ulp, leaves 0.0007 over these arguments), since a sum keeps what does not cancel."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_02067_gb300 import Handle, Problem, build
    build()
    n = 200000
    t = np.random.default_rng(int(abs(lo) + hi)).uniform(lo, hi, n)
    want = np.exp(t.astype(np.longdouble))
    w64 = want.astype(np.float64)
    T = lambda x: torch.as_tensor(np.ascontiguousarray(x)).to(DEV, torch.float64)  # noqa: E731
    h = Handle(0, n, 1)
    r = 2.0 * w64
    prob = Problem(T(np.zeros((n, 1))), T(r), T(np.array([1.7e308])), precision="fp64")
    a = torch.empty(n, dtype=torch.float64, device=DEV)
    h.eot_round(prob, T(t), T(np.zeros(1)), 1.0, None, None, a, None)
    h.close()
    got = r - a.cpu().numpy()
    ulp = np.ldexp(1.0, np.frexp(w64)[1] - 53)
    err = ((got.astype(np.longdouble) - want) / ulp).astype(np.float64)
    assert np.abs(err).max() <= 0.9, np.abs(err).max()
    assert abs(err.mean()) <= 0.02, err.mean()
