"""The batched solver's general sweeps in each of their forms, and its autotuner when
the same shapes come back with other sweeps."""
import numpy as np
import pytest

from oracle import eot_oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture()
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


def batch(given):
    from paper_2504_02067_gb300 import Problem
    ps = [W.uniform_points_problem(30 + k, n, m) for k, (n, m) in enumerate([(40, 300), (520, 260), (1100, 129)])]
    return ps, [Problem(X=t(p["X"], torch.float32), Y=t(p["Y"], torch.float32), r=t(p["r"]), c=t(p["c"]),
                        precision="mixed", cost_scale=O.sqeuclid_scale(p["X"], p["Y"]) if given else 0.0) for p in ps]


@pytest.mark.parametrize("cfg", ["1,1", "2,2", "2,4", "8,4"])
@pytest.mark.parametrize("pgrid", ["0", "1"])
def test_forms(H, cfg, pgrid, monkeypatch):
    """Own elements per thread beyond, at and below a round of the group's threads: each
    problem reaches marginal L1 <= 1e-6 as the oracle measures it."""
    from paper_2504_02067_gb300 import default_params, solve_batched
    monkeypatch.setenv("EOT_BATCH_CFG", cfg)
    monkeypatch.setenv("EOT_PGRID", pgrid)
    ps, probs = batch(False)
    us, vs, st, _ = solve_batched(H, probs, default_params(gamma_i=16.0, gamma_f=256.0))
    assert st == [0] * len(ps)
    for p, u, v in zip(ps, us, vs):
        C = O.sqeuclid_scale(p["X"], p["Y"]) * O.sqeuclid(p["X"], p["Y"])
        assert O.marginal_l1_error(u.cpu().numpy(), v.cpu().numpy(), 256.0, C, p["r"], p["c"]) <= 1e-6


@pytest.mark.parametrize("given", [False, True])
def test_tuned_for_the_sweeps_at_hand(H, given, monkeypatch):
    """A repeated batch is not tuned again; the same shapes on the general sweeps, or at
    a temperature beyond the split's range, are."""
    from paper_2504_02067_gb300 import default_params, solve_batched
    _, probs = batch(given)

    def launches(gamma_f, pgrid="1"):
        monkeypatch.setenv("EOT_PGRID", pgrid)
        l0 = H.launches()
        assert solve_batched(H, probs, default_params(gamma_i=16.0, gamma_f=gamma_f))[2] == [0] * len(probs)
        return H.launches() - l0

    assert launches(256.0) > 1 and launches(256.0) == 1
    assert launches(256.0, "0") > 1 and launches(256.0, "0") == 1
    assert launches(40000.0) > 1 and launches(40000.0) == 1
    assert launches(256.0) == 1
