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


def _calls(jf, S, wl):
    """The calls that end kernels in their last block, with the results of each."""
    X = torch.as_tensor(W.random_state(wl, seed=5, vel=1e-3), device="cuda")
    dt = S.dt_from_cfl(X, 10.0)

    def step():
        Y = X.clone()
        st = S.step(Y, dt)
        return [Y, torch.tensor(st["gmres_iterations"])]

    def si_step():
        Y = X.clone()
        S.si_step(Y, dt)
        return [Y]
    calls = [step, lambda: [S.linear_solve(X, X, dt)[0]], si_step,
             lambda: [S.precond_apply(X, dt, X.to(S.vdtype))], lambda: [S.jv(X, dt, X.to(S.vdtype))[0]]]
    if S.vdtype == torch.float64:
        calls.append(lambda: [S.vjp(X, X, dt, X)[0]])
    return calls


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("cid,n", [(1, (32, 32)), (4, (32, 32, 16))])
def test_the_workspace_is_scratch_between_calls(jf, cid, n, precision):
    """The caller may use the buffer for itself between calls, and two handles may
    take turns on one buffer: same bits as a handle alone (the adjoint, which
    adds atomically, to 1e-9)."""
    wl = W.config(cid, n=n)
    o = jf.default_options(theta=wl.theta, precond=wl.precond, precision=precision)
    S = jf.Solver.from_workload(wl, o)
    T = jf.Solver.from_workload(wl, jf.default_options(theta=wl.theta, precond=1, precision=0, gmres_m=7))
    nbytes = S.workspace.numel()
    if T.workspace.numel() > nbytes:
        S, T = T, S
    base = S.workspace.data_ptr()
    T._check(jf.lib().jfnk_bind(T.h, ctypes.c_void_p(base + (-base) % 256), S.workspace.numel() - 256,
                                ctypes.c_void_p(S.stream.cuda_stream)))
    for k, f in enumerate(_calls(jf, S, wl)):
        ref = f()
        S.workspace.fill_(0x7F)
        again = f()
        _calls(jf, T, wl)[0]()
        third = f()
        for a, b, c in zip(ref, again, third):
            if k == 5:
                assert float((a - b).norm()) < 1e-9 * float(a.norm()) and float((a - c).norm()) < 1e-9 * float(a.norm())
            else:
                assert torch.equal(a, b) and torch.equal(a, c), k
