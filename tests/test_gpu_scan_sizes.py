"""Scan kernels at the sizes where their index arithmetic and launch rules change: every
velocity grid (runs and lanes that do not fill a warp or a CTA), one to three cells (both walls
on one cell), wavefronts of one cell, moving lids and inflow; and scans whose collision-step
Maxwellian is stale, so that the visit's first residual is formed a second time."""
import numpy as np
import pytest
import torch

from paper_2409_01910_gb300 import inputs as I
from paper_2409_01910_gb300 import sgs

pytestmark = pytest.mark.gpu


def state(cells, N, L, seed=1):
    """Distributions around Maxwellians of varying (rho, U, T) and a penalty field of their scale."""
    rng = np.random.default_rng(seed)
    f = np.empty((cells, N, N, N))
    P = np.empty_like(f)
    for j in range(cells):
        M = I.sampled_maxwellian(N, L, 0.8 + 0.4 * rng.random(), tuple(0.3 * (rng.random(3) - 0.5)), 0.9 + 0.6 * rng.random())
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
    st = s.read_status()
    assert st["status"] == 0 and st["visits"] == len(orderings) * p.cells, st
    return f.cpu().numpy().reshape(f0.shape), st


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


# FP64 parity bound of the scans; double-float keeps about 2^-47 per operation
TOL = {sgs.FP64: 1e-12, sgs.FP32: 1e-11}


@pytest.mark.parametrize("precision", [sgs.FP64, sgs.FP32])
@pytest.mark.parametrize("N,J,inflow", [(8, 1, False), (8, 3, True), (12, 2, False), (16, 3, True), (20, 1, True),
                                        (24, 2, False), (28, 2, False), (32, 3, False)])
def test_scan_1d(oracle, N, J, inflow, precision):
    L = 6.0
    kw = dict(eps=0.2, total_mass=1.0, inner_fixed=3, bc_T=(1.0, 1.4))
    if inflow:
        kw.update(bc_kind=(sgs.INFLOW, sgs.DIFFUSE), bc_rho=(1.2, 1.0), bc_u=((0.4, 0.1, 0.0), (0.0, 0.2, 0.0)))
    gp = sgs.Problem(nx=J, nv=N, v_max=L, collision=sgs.BGK, precision=precision, **kw)
    op = oracle.Problem(N=N, L=L, J=J, kernel=oracle.BGK, **kw)
    f0, P0 = state(J, N, L)
    got, st = gpu_scan(gp, f0, P0, [0, 1])
    assert st["inner_iters"] == 2 * 3 * J
    fo = f0.copy()
    nu = np.array([oracle.collision_frequency(op, x) for x in f0])
    for d in (+1, -1):
        oracle.sweep(op, fo, P0, nu, d)
    assert rel(got, fo) <= TOL[precision]


@pytest.mark.parametrize("precision", [sgs.FP64, sgs.FP32])
@pytest.mark.parametrize("N,nx,ny", [(8, 1, 4), (12, 5, 2), (20, 3, 3), (24, 2, 1), (28, 2, 2)])
def test_scan_2d(oracle, N, nx, ny, precision):
    L = 6.0
    kw = dict(eps=0.2, total_mass=1.0, inner_fixed=3, bc_T=(1.0, 1.2))
    ky = dict(bc_T_y=(0.9, 1.1), bc_u_y=((0.0, 0.0, 0.0), (0.4, 0.0, 0.0)))
    gp = sgs.Problem(space_dim=2, nx=nx, ny=ny, nv=N, v_max=L, collision=sgs.BGK, precision=precision, **kw, **ky)
    op = oracle.Problem2D(base=oracle.Problem(N=N, L=L, J=nx, kernel=oracle.BGK, **kw), ny=ny, **ky)
    f0, P0 = state(nx * ny, N, L)
    got, st = gpu_scan(gp, f0, P0, [0, 3, 1, 2])
    assert st["inner_iters"] == 4 * 3 * nx * ny
    fo = f0.copy()
    nu = np.array([oracle.collision_frequency(op.base, x) for x in f0])
    for o in (0, 3, 1, 2):
        oracle.sweep2d(op, fo, P0, nu, o)
    assert rel(got, fo) <= TOL[precision]


@pytest.mark.parametrize("precision", [sgs.FP64, sgs.FP32])
def test_stale_maxwellian_in_tolerance_mode(oracle, precision):
    """Two scans after one collision step: in the second one the stored Maxwellians are not
    those of f. The stop decisions agree with the oracle's (inner_tol far above rounding)."""
    N, J, L = 12, 3, 6.0
    kw = dict(eps=0.2, total_mass=1.0, inner_tol=1e-9, bc_T=(1.0, 1.4))
    gp = sgs.Problem(nx=J, nv=N, v_max=L, collision=sgs.BGK, precision=precision, **kw)
    op = oracle.Problem(N=N, L=L, J=J, kernel=oracle.BGK, **kw)
    f0, P0 = state(J, N, L)
    got, st = gpu_scan(gp, f0, P0, [0, 0])
    fo = f0.copy()
    nu = np.array([oracle.collision_frequency(op, x) for x in f0])
    inner = sum(oracle.sweep(op, fo, P0, nu, +1)["inner_iters"] for _ in range(2))
    assert st["inner_iters"] == inner
    assert rel(got, fo) <= TOL[precision]
