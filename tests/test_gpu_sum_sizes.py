"""Spectral sums at the sizes where their blocks and lane groups change: every velocity grid
(blocks of N/4 outputs, odd ones included), cell counts around the FP64 sum's folded last group
(at most 8 or 16 cells of 32) and several groups, in the three arithmetics."""
import numpy as np
import pytest
import torch

from paper_2409_01910_gb300 import inputs as I
from paper_2409_01910_gb300 import sgs

pytestmark = pytest.mark.gpu


def run(J, N, L, precision, arith=None, sample=None):
    f0 = I.initial_state(J, N, L, T=1.3, noise=2e-2, seed=N + J)
    s = sgs.Solver(sgs.Problem(nx=J, nv=N, v_max=L, precision=precision))
    f = torch.from_numpy(f0.reshape(-1)).cuda()
    Q, P = s.field(), s.field()
    s.collide(f, Q, P, precision=arith)
    assert s.read_status()["status"] == 0
    q = Q.cpu().numpy().reshape(f0.shape)
    return (f0, q) if sample is None else (f0[sample], q[sample])


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("N,J", [(8, 1), (8, 8), (8, 9), (8, 16), (8, 17), (8, 33), (8, 40), (8, 41), (8, 48), (8, 49),
                                 (8, 72), (12, 5), (12, 44), (16, 3), (16, 14)])
def test_fp64_cell_counts(oracle, N, J):
    L = 6.0
    f0, q = run(J, N, L, sgs.FP64)
    qo, _, _ = oracle.collide(oracle.Problem(N=N, L=L, J=J), f0)
    assert rel(q, qo) <= 1e-12  # the FP64 parity bound of the collision step


@pytest.mark.parametrize("arith,tol", [(sgs.FP64, 1e-12), (sgs.DF64, 1e-11), (sgs.FP32, 1e-5)])
@pytest.mark.parametrize("N,J", [(8, 35), (12, 3), (16, 2), (20, 2), (24, 1), (28, 1)])
def test_arithmetics_on_every_grid(oracle, N, J, arith, tol):
    """The bounds of the three arithmetics against the oracle, on the first and last cell."""
    L = 6.0 if N < 24 else 8.0
    f0, q = run(J, N, L, sgs.FP32, arith, sample=[0, J - 1])
    qo, _, _ = oracle.collide(oracle.Problem(N=N, L=L, J=2), np.ascontiguousarray(f0))
    assert rel(q, qo) <= tol
