"""lsms_last_timing's count of kernels equals the kernels of the same application captured as a graph:
FP64 with all pairs stored, with digit products (several right-hand sides' blocks, several runs of
sources, a layout without near pairs), with small and large contour tables, with parts left out; mixed."""
import ctypes

import numpy as np
import pytest

from paper_1407_3868_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1407_3868_gb300 import lsms
    return lsms


def kernels(run):
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    s = torch.cuda.Stream()
    h, graph, count = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t(0)
    assert cu.cuStreamBeginCapture_v2(h, ctypes.c_int(1)) == 0          # thread-local mode
    run(s)
    assert cu.cuStreamEndCapture(h, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(count)) == 0
    total, t = 0, ctypes.c_int()
    for node in nodes:
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)) == 0
        total += t.value == 0
    assert cu.cuGraphDestroy(graph) == 0
    return total


@pytest.mark.parametrize("n,p,nrhs,spread,mixed,flags", [
    (16, 10, 1, 1, False, 0), (120, 6, 1, 1, False, 0), (300, 8, 2, 1, False, 0), (120, 5, 1, 400, False, 0),
    (1000, 15, 5, 1, False, 0), (3000, 15, 1, 1, False, 0), (300, 8, 1, 1, False, 4), (300, 8, 1, 1, False, 8),
    (300, 8, 1, 1, False, 16), (300, 8, 1, 1, True, 2)])
def test_launch_count(L, n, p, nrhs, spread, mixed, flags):
    import torch
    m = inputs.MEDIUM
    h = inputs.widened_half_width(n) * spread
    ctx = L.Context(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"], p, 256, b=inputs.contour_b(2 * h),
                    t_max=141.0, panel_order=16, precision=L.LSMS_MIXED if mixed else L.LSMS_FP64)
    c = inputs.layout(n, -h, h, 4) if spread == 1 else np.stack([np.linspace(-h, h, n), np.full(n, -1.0)], axis=1)
    ctx.set_particles(c)
    x = torch.from_numpy(inputs.random_coefficients(n, p, nrhs, 1)).cuda()
    y = torch.empty_like(x)
    ctx.set_timing(True)
    ctx.apply_dev(x, y, flags)
    torch.cuda.synchronize()
    counted = ctx.last_timing()[2]
    ctx.set_timing(False)
    assert counted == kernels(lambda s: ctx.apply_dev(x, y, flags, stream=s))
    ctx.close()
