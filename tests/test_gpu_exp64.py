"""The FP64 exponential of the FP64 sweeps and of Round (csrc/exp64.cuh), read off
Round's row sums: with one column, v = 0 and C = 0, row i's sum is exp(u_i); with
r_i = 2 exp(u_i) and c larger than every column sum no row or column is scaled, and
a_i = r_i - exp(u_i) is exact (Sterbenz), so r_i - a_i returns exp64's own bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def arguments():
    rng = np.random.default_rng(0)
    edge = [0.0, -0.0, 1e-300, -1e-300, 2.0 ** -20, -(2.0 ** -20), np.nextafter(2.0 ** -20, 0), 1.0, -1.0,
            707.9999, -707.9999, 708.0, -708.0, -708.5, -744.0, -745.2, -745.6, -1e4, -1e300, -np.inf]
    ln2 = np.log(2.0)
    steps = np.arange(-4096, 4097) * ln2 / 2048  # table boundaries and binades
    return np.concatenate([edge, steps, np.nextafter(steps, 10), np.nextafter(steps, -10),
                           rng.uniform(-40, 8, 4000), rng.uniform(-708, 600, 4000),
                           rng.uniform(-1e-3, 1e-3, 1000), rng.uniform(-746, -700, 500)])


def test_exp64_against_libm():
    """Within 2 ulp of numpy's exp everywhere (this exponential errs by at most 1.3
    ulp, numpy's by less than 1 / 2 ulp + its own rounding), within one subnormal
    spacing below 2^-1022, and exactly 0 or 1 where those are the only answers. (The arguments near 708 are few: the column sum stays finite.)"""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_02067_gb300 import Handle, Problem, build
    build()
    t = arguments()
    n = t.size
    want = np.exp(t)
    r = np.where(want > 0, 2.0 * want, 0.0)
    T = lambda x: torch.as_tensor(np.ascontiguousarray(x)).to(DEV, torch.float64)  # noqa: E731
    h = Handle(0, n, 1)
    prob = Problem(T(np.zeros((n, 1))), T(r), T(np.array([1.7e308])), precision="fp64")
    a = torch.empty(n, dtype=torch.float64, device=DEV)
    h.eot_round(prob, T(t), T(np.zeros(1)), 1.0, None, None, a, None)
    got = r - a.cpu().numpy()
    h.close()
    tol = 2.0 * np.spacing(np.where(want > 0, want, 5e-324))
    bad = np.abs(got - want) > tol
    assert not bad.any(), (t[bad][:5], got[bad][:5], want[bad][:5])
    assert (got[t < -745.5] == 0.0).all() and (got[np.abs(t) < 1e-17] == 1.0).all()
