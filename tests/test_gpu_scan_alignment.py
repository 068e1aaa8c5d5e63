"""Scans on fields that start on 8 bytes but not on 16 (contiguous views into larger arrays): the
same bits as on aligned ones."""
import numpy as np
import pytest
import torch

from paper_2409_01910_gb300 import inputs as I
from paper_2409_01910_gb300 import sgs

pytestmark = pytest.mark.gpu


def field(x, odd):
    """x on the GPU, starting at an odd multiple of 8 bytes if asked for."""
    b = torch.zeros(x.size + 2, dtype=torch.float64, device="cuda")
    t = b[1:1 + x.size] if odd else b[:x.size]
    t.copy_(torch.from_numpy(x.reshape(-1)))
    assert t.data_ptr() % 16 == (8 if odd else 0)
    return t


@pytest.mark.parametrize("precision", [sgs.FP64, sgs.FP32])
@pytest.mark.parametrize("N,nx,ny", [(8, 3, 0), (12, 2, 0), (8, 2, 2)])
def test_fields_on_eight_bytes(N, nx, ny, precision):
    kw = dict(space_dim=2, ny=ny, bc_T_y=(0.9, 1.1)) if ny else {}
    p = sgs.Problem(nx=nx, nv=N, v_max=6.0, eps=0.2, bc_T=(1.0, 1.4), collision=sgs.BGK, precision=precision, **kw)
    f0 = I.initial_state(p.cells, N, 6.0, T=1.3, noise=2e-2, seed=3)
    rng = np.random.default_rng(4)
    P0, b0 = (1e-2 * f0 * rng.uniform(-1, 1, f0.shape) for _ in range(2))

    def scan(odd_f, odd_P, odd_b):
        s = sgs.Solver(p)
        f, P, b = field(f0, odd_f), field(P0, odd_P), field(b0, odd_b)
        s.collide(f, s.field(), None)
        for o in (0, 1):
            s.sweep_ordering(f, P, o, rhs=b)
        assert s.read_status()["status"] == 0
        return f

    want = scan(False, False, False)
    for odd in ((True, False, False), (False, True, False), (False, False, True), (True, True, True)):
        assert torch.equal(scan(*odd), want), odd
