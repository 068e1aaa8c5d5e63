"""The scan inside sgs_dc_step: a kernel of its own (1-D), with its own launch shape. Every velocity
grid and number of nodes per thread, one to three cells, the three inner methods; the shapes that
the autotuner times."""
import numpy as np
import pytest
import torch

from paper_2409_01910_gb300 import inputs as I
from paper_2409_01910_gb300 import sgs

pytestmark = pytest.mark.gpu

EPTS = (2, 4, 8, 12, 16, 20, 24, 28, 32)


def shapes(N):
    """The autotuner's candidates: nodes per thread, CTAs per cluster, threads per CTA."""
    out, K = [], N ** 3
    for ept in EPTS:
        for cs in (1, 2, 4, 8, 16):
            tpb = max(160, -(-K // (ept * cs)) + 31 & ~31)
            idle_warp = (tpb - 32) * cs * ept >= K and tpb > 160
            if N % ept == 0 and tpb <= 256 and not idle_warp:
                out.append((ept, cs, tpb))
    return out


def rel(a, b):
    return float((a - b).abs().max() / b.abs().max())


def one_step(N, J, shape=None, **kw):
    """One defect-correction step with one iteration, and the same iteration in FP64."""
    L = 6.0 if N < 24 else 8.0
    p = dict(nx=J, nv=N, v_max=L, bc_T=(1.0, 1.4), inner_fixed=3, **kw)
    f0 = torch.from_numpy(I.initial_state(J, N, L, T=1.2, noise=2e-2, seed=N).reshape(-1)).cuda()
    out = []
    for precision in (sgs.FP32, sgs.FP64):
        s = sgs.Solver(sgs.Problem(precision=precision, **p))
        f, Q, P = f0.clone(), s.field(), s.field()
        if precision == sgs.FP32:
            if shape:
                s.set_sweep_shape(*shape)
            s.dc_step(f, Q, P, 1)
        else:
            s.iterate(f, Q, P)
        st = s.read_status()
        assert st["status"] == 0 and st["inner_iters"] == 2 * 3 * J and st["visits"] == 2 * J, st
        out.append(f)
    return out[0], out[1], rel(out[1], f0)


# The backward scan's collision step is the reference's plus increments summed in FP32: rounding
# of 1e-6 of the change of f (the FP32 sums' error against FP64 is below 2e-6 of Q), which is at
# most a few tenths here.
@pytest.mark.parametrize("N,J", [(8, 1), (8, 3), (12, 2), (16, 3), (20, 1), (24, 2), (28, 1), (32, 2)])
def test_every_grid(N, J):
    f, want, change = one_step(N, J, eps=0.2)
    assert rel(f, want) <= 2e-6 * max(change, 0.1)


@pytest.mark.parametrize("N,ept", [(N, e) for N in (8, 12, 16, 20, 24, 28, 32) for e in EPTS if N % e == 0 and N ** 3 <= e * 4096])
def test_every_number_of_nodes_per_thread(N, ept):
    shape = next(s for s in shapes(N) if s[0] == ept)
    f, want, change = one_step(N, 2, shape, eps=0.2)
    assert rel(f, want) <= 2e-6 * max(change, 0.1)


@pytest.mark.parametrize("method,eps", [(sgs.FP, 0.5), (sgs.PFP_RELAX, 0.2), (sgs.PFP_RELAX, 0.02)])
def test_inner_methods(method, eps):
    f, want, change = one_step(12, 3, eps=eps, inner_method=method)
    assert rel(f, want) <= 2e-6 * max(change, 0.1)


@pytest.mark.parametrize("N,precision,collision,ny", [(16, sgs.FP64, sgs.MAXWELL, 0), (16, sgs.FP32, sgs.MAXWELL, 0),
                                                      (12, sgs.FP32, sgs.BGK, 0), (8, sgs.FP32, sgs.MAXWELL, 2)])
def test_autotuner_times_what_runs(N, precision, collision, ny):
    """One candidate for each launch of the scans, and one for each shape of the scan inside sgs_dc_step
    where the handle has it; what is reported can be given to another handle."""
    kw = dict(space_dim=2, ny=ny) if ny else {}
    p = sgs.Problem(nx=2, nv=N, v_max=6.0, eps=0.2, collision=collision, precision=precision, inner_fixed=2, **kw)
    s = sgs.Solver(p)
    f = torch.from_numpy(I.initial_state(p.cells, N, 6.0, T=1.2, noise=1e-2, seed=1).reshape(-1)).cuda()
    P = s.field()
    s.collide(f, s.field(), P)
    t = s.autotune(f, P)
    scans = len({x[1:] for x in shapes(N)})
    dc = precision == sgs.FP32 and collision != sgs.BGK and not ny
    assert t["candidates"] == scans + (len(shapes(N)) if dc else 0)
    assert s.sweep_shape() in shapes(N)
    o = sgs.Solver(p)
    o.set_sweep_shape(*s.sweep_shape())
    assert o.sweep_shape() == s.sweep_shape()
