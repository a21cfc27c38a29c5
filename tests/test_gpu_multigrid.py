"""The multigrid kernels against the oracle on the shapes where their
dispatch changes: rows too short for vectors, rows that fill them, extents
that run out in x before y and z (levels in natural order), grids whose
coarse levels fit one kernel from the start, 2D levels of whole tiles (one tile
wide, too), and cycles without pre- or
post-smoothing.  FP64 applies agree to 1e-10 (the operator is fixed and
linear; only the order of its sums differs), FP32 ones to 1e-4 (the bound of
the full-size parity tests)."""
import ctypes
import math

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


SHAPES = [(1, (4, 64)), (1, (64, 4)), (2, (8, 512)), (2, (256, 256)), (2, (128, 128)), (2, (32, 1024)), (1, (256, 128)), (3, (4, 8, 64)), (3, (64, 64, 16)),
          (4, (8, 32, 64)), (4, (64, 64, 64)), (4, (128, 16, 8))]


@pytest.mark.parametrize("cid,n", SHAPES)
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (0, 2), (1, 0)])
def test_apply_matches_the_oracle(jf, cid, n, precision, nu):
    wl = W.config(cid, n=n, mach=1e-2 if cid == 3 else None)
    X = W.random_state(wl, seed=7, vel=1e-3)
    P = D.Problem.from_workload(wl)
    dt = D.cfl_dt(P, X, 10.0)
    op = J.Options(precond=wl.precond, mg_cycles=2, mg_nu1=nu[0], mg_nu2=nu[1])
    sc = J.scaling(P, X, op)
    v = torch.as_tensor(W.random_vector(wl, seed=8))
    ref = PC.apply(PC.setup(P, X, dt, op), v, sc)
    o = jf.default_options(theta=wl.theta, precond=wl.precond, mg_cycles=2, mg_nu1=nu[0], mg_nu2=nu[1],
                           precision=precision)
    S = jf.Solver.from_workload(wl, o)
    w = S.precond_apply(torch.as_tensor(X, device="cuda"), dt, v.to("cuda", S.vdtype)).double().cpu()
    err = float((w - ref).norm() / ref.norm())
    assert err < (1e-4 if precision else 1e-10), err


@pytest.mark.parametrize("cid,n", [(1, (32, 16)), (4, (16, 16, 8))])
def test_unaligned_vectors_take_the_general_transforms(jf, cid, n):
    """Vectors that start off a 16-byte boundary are applied to by the
    transforms that move single values; both agree to the FP32 bound of the
    applies, and neither writes outside its output."""
    wl = W.config(cid, n=n)
    X = torch.as_tensor(W.random_state(wl, seed=3, vel=1e-3), device="cuda")
    S = jf.Solver.from_workload(wl, jf.default_options(theta=wl.theta, precond=wl.precond, precision=jf.MIXED))
    dt = S.dt_from_cfl(X, 10.0)
    v = torch.as_tensor(W.random_vector(wl, seed=4), device="cuda").float()
    ref = S.precond_apply(X, dt, v)
    buf = torch.full((S.nvec + 2,), 7.0, device="cuda")
    vin = torch.cat([v.new_zeros(1), v])[1:]
    S.precond_apply(X, dt, vin, out=buf[1:-1])
    assert float(buf[0]) == 7.0 and float(buf[-1]) == 7.0
    assert float((buf[1:-1] - ref).norm() / ref.norm()) < 1e-4
    assert float((S.precond_apply(X, dt, v) - ref).norm()) == 0.0


@pytest.mark.parametrize("cid,n", [(1, (128, 64)), (4, (32, 32, 32))])
@pytest.mark.parametrize("precision", [0, 1])
def test_the_output_may_overlap_the_input(jf, cid, n, precision):
    """An apply in place, and one whose output starts inside its input (and the
    other way round), give what separate vectors give: to the FP32 bound where
    the transforms differ, else the same bits."""
    wl = W.config(cid, n=n)
    X = torch.as_tensor(W.random_state(wl, seed=3, vel=1e-3), device="cuda")
    S = jf.Solver.from_workload(wl, jf.default_options(theta=wl.theta, precond=wl.precond, precision=precision))
    dt = S.dt_from_cfl(X, 10.0)
    v = torch.as_tensor(W.random_vector(wl, seed=4), device="cuda").to(S.vdtype)
    ref = S.precond_apply(X, dt, v)
    nc = S.nvec // (2 + wl.ndim)
    for shift in (0, 4, -4, nc, -2 * nc, S.nvec):
        buf = torch.zeros(S.nvec + abs(shift), dtype=S.vdtype, device="cuda")
        i, o = max(-shift, 0), max(shift, 0)
        buf[i:i + S.nvec] = v
        w = S.precond_apply(X, dt, buf[i:i + S.nvec], out=buf[o:o + S.nvec])
        err = float((w - ref).norm() / ref.norm())
        assert err < (1e-4 if precision and shift not in (0, S.nvec) else 1e-300), (shift, err)


# mean relative errors of the density, energy and velocity rows of an FP32 apply
# that forms and divides by the diagonal block in every sweep (four inputs each)
DIVIDED = [(1, (512, 256), 0.5, 1, (1.108e-7, 8.819e-8, 2.223e-6)), (2, (256, 256), 0.5, 2, (1.703e-7, 1.620e-7, 9.869e-7)),
           (2, (512, 512), 1.0, 1, (2.421e-7, 2.270e-7, 2.597e-6)), (3, (64, 64, 64), 0.5, 2, (1.113e-7, 8.864e-8, 1.947e-7)),
           (4, (64, 64, 64), 0.5, 2, (1.068e-7, 9.871e-8, 1.718e-7))]


@pytest.mark.parametrize("cid,n,theta,nu,bound", DIVIDED)
def test_inverse_blocks_lose_no_digit_of_an_fp32_apply(jf, cid, n, theta, nu, bound):
    """The rounded inverse diagonal blocks leave no larger error in an FP32 apply
    (against the FP64 handle on the same vector) than dividing did."""
    sums = [0.0, 0.0, 0.0]
    for seed in range(4):
        wl = W.config(cid, n=n)
        X = torch.as_tensor(W.random_state(wl, seed=20 + seed, vel=1e-3), device="cuda")
        v = torch.as_tensor(W.random_vector(wl, seed=40 + seed), device="cuda").float()
        w = []
        for precision in (1, 0):
            S = jf.Solver.from_workload(wl, jf.default_options(theta=theta, precond=wl.precond, precision=precision,
                                                               mg_nu1=nu, mg_nu2=nu))
            w.append(S.precond_apply(X, S.dt_from_cfl(X, 0.2 * max(n)), v.to(S.vdtype)).double())
        nc = v.numel() // (2 + wl.ndim)
        for k, (a, b) in enumerate(((0, nc), (nc, 2 * nc), (2 * nc, v.numel()))):
            sums[k] += float((w[0] - w[1])[a:b].norm() / w[1][a:b].norm()) / 4
    assert all(e <= b for e, b in zip(sums, bound)), (sums, bound)


@pytest.mark.parametrize("cid,n,mass,time", [(1, (64, 64), -90, 60), (3, (16, 16, 16), -90, 60), (2, (64, 64), -20, 20),
                                             (1, (64, 64), 40, -60)])
def test_an_fp32_apply_does_not_depend_on_the_units(jf, cid, n, mass, time):
    """Density times 2^mass, lengths and times times 2^time (velocities and
    energies unchanged): every operation scales by a power of two, so the apply,
    which has the dimension of a time, scales by 2^time bit for bit.  dt / rho
    is far beyond the range of a float in the first two cases."""
    wl = W.config(cid, n=n, mach=1e-2 if cid == 3 else None)
    X = torch.as_tensor(W.random_state(wl, seed=6, vel=1e-3), device="cuda")
    v = torch.as_tensor(W.random_vector(wl, seed=9), device="cuda").float()
    o = jf.default_options(theta=wl.theta, precond=wl.precond, precision=jf.MIXED)
    S = jf.Solver.from_workload(wl, o)
    dt = 2.0 ** round(math.log2(S.dt_from_cfl(X, 10.0)))
    ref = S.precond_apply(X, dt, v)
    m, t = 2.0 ** mass, 2.0 ** time
    Y = X.clone()
    Y[:X.numel() // (2 + wl.ndim)] *= m
    T = jf.Solver(wl.ndim, wl.n, [q * t for q in wl.lo], [q * t for q in wl.hi], wl.bc, wl.gamma, wl.energy_form,
                  [q / t for q in wl.g], wl.K0 * m * t, wl.chi_exp, o)
    w = T.precond_apply(Y, dt * t, v)
    assert bool(torch.isfinite(w).all()) and torch.equal(w.double(), ref.double() * t)


def _against_the_oracle(jf, cid, n, precision, nu, cluster=None):
    wl = W.config(cid, n=n, mach=1e-2 if cid == 3 else None)
    X = W.random_state(wl, seed=7, vel=1e-3)
    P = D.Problem.from_workload(wl)
    dt = D.cfl_dt(P, X, 10.0)
    op = J.Options(precond=wl.precond, mg_cycles=2, mg_nu1=nu[0], mg_nu2=nu[1])
    v = torch.as_tensor(W.random_vector(wl, seed=8))
    ref = PC.apply(PC.setup(P, X, dt, op), v, J.scaling(P, X, op))
    S = jf.Solver.from_workload(wl, jf.default_options(theta=wl.theta, precond=wl.precond, mg_cycles=2, mg_nu1=nu[0],
                                                       mg_nu2=nu[1], precision=precision))
    if cluster is not None:
        f = getattr(jf.lib(), "_Z23jfnk_handle_set_clusterP11jfnk_handlei")
        f.restype, f.argtypes = None, [ctypes.c_void_p, ctypes.c_int]
        f(S.h, cluster)
    w = S.precond_apply(torch.as_tensor(X, device="cuda"), dt, v.to("cuda", S.vdtype)).double().cpu()
    err = float((w - ref).norm() / ref.norm())
    assert err < (1e-4 if precision else 1e-10), err


@pytest.mark.parametrize("cid,n", [(2, (4, 131072)), (1, (4, 131072)), (4, (4, 256, 2048))])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nu", [(2, 2), (0, 2)])
def test_levels_in_natural_order_above_the_cluster(jf, cid, n, precision, nu):
    """x runs out on a level of 32,768 cells, too many for the cluster kernel in
    either precision: smoother, residual and transfers of levels in natural
    order run as kernels of their own."""
    _against_the_oracle(jf, cid, n, precision, nu)


@pytest.mark.parametrize("cid,n", [(1, (64, 4)), (2, (128, 128)), (2, (8, 512)), (4, (32, 32, 32)), (4, (128, 16, 8)),
                                   (3, (4, 8, 64))])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nu", [(2, 2), (1, 0), (0, 2)])
@pytest.mark.parametrize("cluster", [0, 8])
def test_devices_with_smaller_clusters_or_none(jf, cid, n, precision, nu, cluster):
    """A cluster of eight blocks, or every level down to the single cell by
    kernels of its own, give the same apply."""
    _against_the_oracle(jf, cid, n, precision, nu, cluster)
