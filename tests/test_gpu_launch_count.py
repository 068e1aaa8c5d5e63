"""sgs_launch_count against the kernel nodes of a captured call, at cell counts where the FP64 sum
is one kernel or two (a last lane group of at most 16 cells is summed by one of its own)."""
import ctypes as C

import pytest
import torch

from paper_2409_01910_gb300 import inputs as I
from paper_2409_01910_gb300 import sgs

pytestmark = pytest.mark.gpu


def kernel_nodes(call):
    """Kernel nodes of the graph that `call` captures to."""
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    cuda = C.CDLL("libcuda.so.1")
    raw, n = C.c_void_p(g.raw_cuda_graph()), C.c_size_t(0)
    assert cuda.cuGraphGetNodes(raw, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cuda.cuGraphGetNodes(raw, nodes, C.byref(n)) == 0
    kinds = []
    for x in nodes:
        t = C.c_int(-1)
        assert cuda.cuGraphNodeGetType(C.c_void_p(x), C.byref(t)) == 0
        kinds.append(t.value)
    return kinds.count(0)  # CU_GRAPH_NODE_TYPE_KERNEL


@pytest.mark.parametrize("cells", [8, 16, 17, 32, 40, 48, 49, 64, 72])
@pytest.mark.parametrize("precision,arith", [(sgs.FP64, sgs.FP64), (sgs.FP32, sgs.FP64), (sgs.FP32, sgs.FP32),
                                             (sgs.FP32, sgs.DF64)])
def test_collide_launches(cells, precision, arith):
    s = sgs.Solver(sgs.Problem(nx=cells, nv=8, v_max=6.0, precision=precision))
    f = torch.from_numpy(I.initial_state(cells, 8, 6.0, T=1.2, seed=1).reshape(-1)).cuda()
    Q, P = s.field(), s.field()
    s.collide(f, Q, P, precision=arith)  # sets the kernels' attributes outside the capture
    before = s.launch_count()
    nodes = kernel_nodes(lambda: s.collide(f, Q, P, precision=arith))
    assert s.launch_count() - before == nodes


@pytest.mark.parametrize("cells", [17, 40, 72])
def test_autotuned_sum_is_what_runs(cells):
    """Blocks of the reported decomposition: per work unit one for every `sum_warps` lane groups, and
    one for a folded last group."""
    s = sgs.Solver(sgs.Problem(nx=cells, nv=8, v_max=6.0, inner_fixed=1))
    f = torch.from_numpy(I.initial_state(cells, 8, 6.0, T=1.2, seed=1).reshape(-1)).cuda()
    P = s.field()
    s.collide(f, s.field(), P)
    t = s.autotune(f, P)
    groups = -(-cells // 32)
    folded = cells - 32 * (groups - 1) <= 16
    rest = groups - folded
    assert t["sum_blocks"] == t["sum_units"] * (-(-rest // t["sum_warps"]) + folded)
    assert t["sum_warps"] <= max(1, rest)
