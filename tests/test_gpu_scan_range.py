"""Scans at the ends of the range of states: gases that move at many thermal speeds along the
walls (the factors of their Maxwellian reach exp(U^2 / 2T), whose square leaves FP32) and thin ones
(the squares of their residuals sink below it). The stop decisions of the inner iteration agree
with the oracle's (the tolerance is far above rounding)."""
import numpy as np
import pytest
import torch

from paper_2409_01910_gb300 import inputs as I
from paper_2409_01910_gb300 import sgs

pytestmark = pytest.mark.gpu


def state(cells, N, L, U, T, seed=1):
    rng = np.random.default_rng(seed)
    f = np.empty((cells, N, N, N))
    P = np.empty_like(f)
    for j in range(cells):
        u = tuple(np.asarray(U) + 0.05 * np.sqrt(T) * rng.uniform(-1, 1, 3))
        M = I.sampled_maxwellian(N, L, 0.9 + 0.2 * rng.random(), u, T * (0.95 + 0.1 * rng.random()))
        d = M * 1e-2 * rng.uniform(-1, 1, size=M.shape)
        f[j], P[j] = M + d, 0.3 * d
    return f, P


def gpu_scan(p, f0, P0, orderings):
    s = sgs.Solver(p)
    f = torch.from_numpy(f0.reshape(-1).copy()).cuda()
    P = torch.from_numpy(P0.reshape(-1).copy()).cuda()
    s.collide(f, s.field(), None)
    for o in orderings:
        s.sweep_ordering(f, P, o)
    return f.cpu().numpy().reshape(f0.shape), s.read_status()


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def tol(U, T):
    """The parity bound of the scans, 1e-12 for a gas at rest, times what a temperature loses to
    rounding when it is formed from the raw moments of a moving one."""
    return 1e-12 * (1.0 + np.dot(U, U) / (3.0 * T))


@pytest.mark.parametrize("U", [(0.2, 4.0, 0.0), (0.2, 5.0, 0.0), (0.1, 0.2, 5.4)])
def test_fast_along_the_walls_1d(oracle, U):
    N, J, L, T = 32, 2, 8.0, 0.25
    kw = dict(eps=0.2, total_mass=1.0, inner_tol=1e-9, bc_kind=(sgs.INFLOW, sgs.INFLOW), bc_u=(U, U), bc_T=(T, T))
    op = oracle.Problem(N=N, L=L, J=J, kernel=oracle.BGK, **kw)
    f0, P0 = state(J, N, L, U, T)
    got, st = gpu_scan(sgs.Problem(nx=J, nv=N, v_max=L, collision=sgs.BGK, **kw), f0, P0, [0, 1])
    fo = f0.copy()
    nu = np.array([oracle.collision_frequency(op, x) for x in f0])
    inner = sum(oracle.sweep(op, fo, P0, nu, d)["inner_iters"] for d in (+1, -1))
    assert st["status"] == 0 and st["inner_iters"] == inner, (st, inner)
    assert rel(got, fo) <= tol(U, T)


@pytest.mark.parametrize("precision", [sgs.FP64, sgs.FP32])
@pytest.mark.parametrize("N,L,T,U", [(16, 6.0, 0.3, (3.0, 0.0, 0.0)), (24, 6.0, 0.2, (3.0, 1.5, 0.5)),
                                     (32, 8.0, 0.25, (5.0, 0.5, 0.5))])
def test_cold_fast_gas(oracle, N, L, T, U, precision):
    """Newton's closing step is taken with an FP32 direction from raw moments, whose rounding grows
    with the speed, as that of an evaluation does."""
    J = 3
    kw = dict(eps=0.05, total_mass=1.0, inner_fixed=4, bc_kind=(sgs.INFLOW, sgs.INFLOW), bc_u=(U, U), bc_T=(T, T))
    op = oracle.Problem(N=N, L=L, J=J, kernel=oracle.BGK, **kw)
    f0, P0 = state(J, N, L, U, T)
    got, st = gpu_scan(sgs.Problem(nx=J, nv=N, v_max=L, collision=sgs.BGK, precision=precision, **kw), f0, P0, [0, 1])
    assert st["status"] == 0 and st["inner_iters"] == 2 * 4 * J, st
    fo = f0.copy()
    nu = np.array([oracle.collision_frequency(op, x) for x in f0])
    for d in (+1, -1):
        oracle.sweep(op, fo, P0, nu, d)
    assert rel(got, fo) <= (1.0 if precision == sgs.FP64 else 10.0) * tol(U, T)


def test_fast_along_the_walls_2d(oracle):
    N, nx, ny, L, T, U = 32, 2, 1, 8.0, 0.25, (0.1, 0.2, 5.0)
    kw = dict(eps=0.2, total_mass=1.0, inner_tol=1e-9, bc_kind=(sgs.INFLOW, sgs.INFLOW), bc_u=(U, U), bc_T=(T, T))
    ky = dict(bc_kind_y=(sgs.INFLOW, sgs.INFLOW), bc_u_y=(U, U), bc_T_y=(T, T))
    op = oracle.Problem2D(base=oracle.Problem(N=N, L=L, J=nx, kernel=oracle.BGK, **kw), ny=ny, **ky)
    f0, P0 = state(nx * ny, N, L, U, T)
    gp = sgs.Problem(space_dim=2, nx=nx, ny=ny, nv=N, v_max=L, collision=sgs.BGK, **kw, **ky)
    got, st = gpu_scan(gp, f0, P0, [0])
    fo = f0.copy()
    nu = np.array([oracle.collision_frequency(op.base, x) for x in f0])
    inner = oracle.sweep2d(op, fo, P0, nu, 0)["inner_iters"]
    assert st["status"] == 0 and st["inner_iters"] == inner, (st, inner)
    assert rel(got, fo) <= tol(U, T)


@pytest.mark.parametrize("precision,rho", [(sgs.FP64, 1e-15), (sgs.FP64, 1e-10), (sgs.FP32, 1e-7)])
def test_thin_gas(oracle, precision, rho):
    """rho times the state of a gas of density one, at rho times its Knudsen number, is rho times
    its solution after the same number of updates."""
    N, J, L, T, U = 12, 3, 6.0, 1.0, (0.2, 0.1, 0.0)
    kw = dict(total_mass=1.0, bc_kind=(sgs.INFLOW, sgs.INFLOW), bc_u=(U, U), bc_T=(T, T))
    op = oracle.Problem(N=N, L=L, J=J, kernel=oracle.BGK, eps=0.2, inner_tol=1e-9, **kw)
    gp = sgs.Problem(nx=J, nv=N, v_max=L, collision=sgs.BGK, precision=precision, eps=0.2 * rho, inner_tol=1e-9 * rho,
                     bc_rho=(rho, rho), **kw)
    f0, P0 = state(J, N, L, U, T)
    got, st = gpu_scan(gp, rho * f0, rho * rho * P0, [0, 1])  # P is quadratic in f
    fo = f0.copy()
    nu = np.array([oracle.collision_frequency(op, x) for x in f0])
    inner = sum(oracle.sweep(op, fo, P0, nu, d)["inner_iters"] for d in (+1, -1))
    assert st["status"] == 0 and st["inner_iters"] == inner, (st, inner)
    assert rel(got / rho, fo) <= (1e-12 if precision == sgs.FP64 else 1e-11)
