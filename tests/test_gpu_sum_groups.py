"""FP32 and FP64 sums over several lane groups of 32 cells, whole and ragged, one or more of them to a
block: every cell against the double-float evaluation of the same state."""
import pytest
import torch

from paper_2409_01910_gb300 import inputs as I
from paper_2409_01910_gb300 import sgs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,J", [(8, 31), (8, 33), (8, 64), (8, 97), (8, 160), (12, 65), (12, 129), (16, 96), (20, 40),
                                 (20, 65), (24, 65)])
def test_every_group(N, J):
    L = 6.0 if N < 24 else 8.0
    s = sgs.Solver(sgs.Problem(nx=J, nv=N, v_max=L, precision=sgs.FP32))
    f = torch.from_numpy(I.initial_state(J, N, L, T=1.3, noise=2e-2, seed=N + J).reshape(-1)).cuda()
    Q = {a: s.field() for a in (sgs.FP32, sgs.FP64, sgs.DF64)}
    for a, q in Q.items():
        s.collide(f, q, None, precision=a)
    assert s.read_status()["status"] == 0
    per_cell = {a: q.reshape(J, -1) for a, q in Q.items()}
    scale = per_cell[sgs.DF64].abs().max()
    # the bounds of the arithmetics against the oracle, 1e-5 and 1e-12, with the double-float one's 1e-11
    for a, tol in ((sgs.FP32, 1e-5), (sgs.FP64, 2e-11)):
        assert float(((per_cell[a] - per_cell[sgs.DF64]).abs().max(dim=1).values / scale).max()) <= tol
