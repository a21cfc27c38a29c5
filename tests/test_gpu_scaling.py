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


@pytest.mark.parametrize("a1,a2", [(-1e-2, 1.0), (1e-5, -1.0), (-0.5, -0.5), (0.0, 0.0)])
def test_alphas_that_set_no_floor_leave_the_velocity(jf, a1, a2):
    """L_u = rho_f max(|u|, alpha1 c_s), R_u = max(|u|, alpha2 c_s): with an alpha
    that is not positive the velocity alone is left."""
    S, X = _solver(jf, alpha1=a1, alpha2=a2)
    n = (16, 32)
    rho, e, u, w = (X[k * 512:(k + 1) * 512].view(n) for k in range(4))
    cs = torch.sqrt(5.0 / 3.0 * (2.0 / 3.0) * e)
    L, R, _ = S.scaling(X)
    for c, q in ((0, u), (1, w)):
        face = lambda f: 0.5 * (f + f.roll(1, 1 - c))  # noqa: E731
        for out, alpha, scale in ((L, a1, face(rho)), (R, a2, torch.ones_like(rho))):
            ref = scale * torch.maximum(q.abs(), alpha * face(cs))
            got = out[(2 + c) * 512:(3 + c) * 512].view(n)
            assert float(((got - ref) / ref).abs().max()) < 1e-14
