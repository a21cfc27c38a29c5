"""What the workspace held before a call does not enter its results: applies and
steps on a workspace full of NaN, and after a vector that held one."""
import ctypes

import pytest
import torch

import workloads as W
from oracle import discretization as D
from oracle import jfnk as J
from oracle import precond as PC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jf():
    import paper_1512_03662_gb300 as jf
    jf.lib()
    return jf


def _fill(S, jf, byte=0xFF):
    """Every byte of the workspace set (0xFF: NaN in both precisions), then bound again."""
    S.workspace.fill_(byte)
    base = S.workspace.data_ptr()
    nbytes = S.workspace.numel() - 256
    S._check(jf.lib().jfnk_bind(S.h, ctypes.c_void_p(base + (-base) % 256), nbytes,
                                ctypes.c_void_p(S.stream.cuda_stream)))


# extents that reach one cell above the levels that one kernel takes together, and ones that do not
THIN = [(4, (128, 128, 4)), (4, (256, 256, 4)), (3, (256, 256, 4)), (4, (4, 128, 128)), (2, (4096, 4)), (1, (64, 64)),
        (2, (256, 256)), (4, (32, 32, 32))]


@pytest.mark.parametrize("cid,n", THIN)
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (0, 2)])
def test_apply_does_not_read_what_the_workspace_held(jf, cid, n, precision, nu):
    """FP64 applies agree with the oracle to 1e-10 and FP32 ones to 1e-4 (the
    bounds of the multigrid tests), on a workspace of NaN and after an apply
    to a vector of NaN."""
    wl = W.config(cid, n=n, mach=1e-2 if cid == 3 else None)
    X = W.random_state(wl, seed=7, vel=1e-3)
    P = D.Problem.from_workload(wl)
    dt = D.cfl_dt(P, X, 10.0)
    op = J.Options(precond=wl.precond, mg_cycles=2, mg_nu1=nu[0], mg_nu2=nu[1])
    v = torch.as_tensor(W.random_vector(wl, seed=8))
    ref = PC.apply(PC.setup(P, X, dt, op), v, J.scaling(P, X, op))
    o = jf.default_options(theta=wl.theta, precond=wl.precond, mg_cycles=2, mg_nu1=nu[0], mg_nu2=nu[1],
                           precision=precision)
    S = jf.Solver.from_workload(wl, o)
    _fill(S, jf)
    Xg, vg = torch.as_tensor(X, device="cuda"), v.to("cuda", S.vdtype)
    for held in ("workspace", "vector"):
        if held == "vector":
            S.precond_apply(Xg, dt, torch.full_like(vg, float("nan")))
        w = S.precond_apply(Xg, dt, vg).double().cpu()
        err = float((w - ref).norm() / ref.norm())
        assert err < (1e-4 if precision else 1e-10), (held, err)
