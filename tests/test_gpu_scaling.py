"""The scaling's edges: states without a finite norm and alphas that set no floor."""
import math

import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jf():
    import paper_1512_03662_gb300 as jf
    jf.lib()
    return jf


def _solver(jf, cid=1, n=(32, 16), **kw):
    wl = W.config(cid, n=n)
    S = jf.Solver.from_workload(wl, jf.default_options(theta=wl.theta, precond=0, **kw))
    return S, torch.as_tensor(W.random_state(wl, seed=2, vel=1e-2), device="cuda")


@pytest.mark.parametrize("row", [0, 1])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), 0.0])
def test_a_state_without_a_finite_norm_says_so(jf, row, value):
    """||R^-1 X|| and the step of the Jacobian-free product are NaN when one
    density or energy is NaN, infinite or zero (R is X there: NaN / NaN,
    infinity times zero), and so is every entry of the product."""
    S, X = _solver(jf)
    v = torch.ones(S.nvec, dtype=torch.float64, device="cuda")
    nc = S.nvec // 4
    X[row * nc + 37] = value
    assert math.isnan(S.scaling(X)[2])
    Jv, delta = S.jv(X, 1e-3, v)
    assert math.isnan(delta) and bool(torch.isnan(Jv).all())
