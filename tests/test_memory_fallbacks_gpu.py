"""The digit products' tables, sequences and images are memory the library can do without.  With no room
for them (the library's own limits, lowered from here: no GPU is run out of memory) the FP64 kernels that
need none take over: all pairs, row ranges, the near field of the boxes, the contour products.  When
another request fails while they are held, they are given back and the request is granted: a solve, the
applications and solves of a batch.  Inside a stream capture nothing is allocated.

Against the oracle: 1e-11 in the scaled norm for translations (as tests/test_translate_f64_tc_gpu.py), 1e-10
for the other FP64 steps and between two FP64 paths (the oracle's tolerance for FP64 steps)."""
import ctypes

import numpy as np
import pytest

from oracle import lsms_oracle as O
from paper_1407_3868_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL_T, TOL = 1e-11, 1e-10
NONE = 2 ** 64 - 1


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1407_3868_gb300 import lsms
    return lsms


def limits(ctx, optional=NONE, required=NONE):
    f = ctx.lib._Z13memory_limitsP8lsms_ctxmm          # the library's own hook
    f.restype = None
    f(ctx.h, ctypes.c_size_t(optional), ctypes.c_size_t(required))


def usable(ctx):
    f = ctx.lib._Z12f64tc_usablePK8lsms_ctx
    f.restype = ctypes.c_bool
    return f(ctx.h)


def context(L, n, p, precision=0, **kw):
    m = dict(inputs.MEDIUM, **kw)
    h = inputs.widened_half_width(n)
    ctx = L.Context(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"], p, 384, b=inputs.contour_b(2 * h),
                    t_max=141.0, panel_order=16, precision=precision)
    return ctx, inputs.layout(n, -h, h, 5), m, O.order_scale(p, m["k2"], m["radius"])


def rel(a, b, hs):
    return np.linalg.norm((a - b) / hs) / np.linalg.norm(b / hs)


@pytest.mark.parametrize("n,p,medium", [(300, 10, {}), (50, 7, {}),
                                        # mostly near pairs, too many to store them all: no limit needed
                                        (400, 12, dict(k1=0.04, k2=0.06, k3=0.05, kp=0.05))])
def test_without_optional_memory(L, n, p, medium):
    import torch
    ctx, c, m, hs = context(L, n, p, **medium)
    if not medium:
        limits(ctx, optional=0)
    ctx.set_particles(c)
    assert not usable(ctx)
    x = inputs.random_coefficients(n, p, 2, 3) / hs
    a = ctx.translate(x)
    rows = [0, 1, n // 2, n - 1]
    for r in range(2):
        assert rel(a[r][rows], O.translate(c, x[r], m["k2"], p, rows), hs) <= TOL_T
    xd = torch.from_numpy(x).cuda()
    y = torch.zeros((2, 20, 2 * p + 1), dtype=torch.complex128, device="cuda")
    ctx.apply_rows_dev(xd, y, 17, 37, L.APPLY_ALPHA | L.APPLY_NO_REFLECTION)
    torch.cuda.synchronize()
    for r in range(2):
        assert rel(y[r].cpu().numpy(), a[r, 17:37], hs) <= TOL_T
    if medium:
        ctx.close()
        return
    lam, wt = ctx.contour()
    pr = O.Problem(O.Medium(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"]), p, c, lam, wt)
    assert rel(ctx.apply(x[:1], L.APPLY_ALPHA | L.APPLY_NO_TRANSLATION)[0], pr.reflection(x[0]), hs) <= TOL
    ctx.set_fmm(4.0)
    b = ctx.translate(x)
    for r in range(2):
        assert rel(b[r], a[r], hs) <= TOL
    ctx.close()


def test_several_blocks_of_right_hand_sides(L):
    n, p = 1000, 15                                     # two right-hand sides' digit images at a time
    ctx, c, m, hs = context(L, n, p)
    ctx.set_particles(c)
    assert usable(ctx)
    x = inputs.random_coefficients(n, p, 5, 9) / hs
    a = ctx.translate(x)
    rows = [0, 130, n - 1]
    for r in range(5):
        assert rel(a[r][rows], O.translate(c, x[r], m["k2"], p, rows), hs) <= TOL_T
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_solve_takes_optional_memory_back(L, precision):
    n, p = 200, 8
    ctx, c, _, hs = context(L, n, p, precision)
    ctx.set_particles(c)
    src = [[0.0, 1.0], [1.0, 1.0]]
    ref, _ = ctx.solve(src, tol=1e-10, maxiter=600)
    assert usable(ctx)                                  # a mixed solve's FP64 residual has stored the sequences
    ctx.close()
    ctx, c, _, _ = context(L, n, p, precision)
    ctx.set_particles(c)
    assert usable(ctx) == (precision == 0)              # a mixed context holds none before
    ctx.translate(np.ones((1, n, 2 * p + 1), dtype=complex))
    assert usable(ctx)
    limits(ctx, required=0)
    beta, _ = ctx.solve(src, tol=1e-10, maxiter=600)
    assert not usable(ctx)
    for r in range(2):
        assert np.linalg.norm((beta[r] - ref[r]) * hs) <= 1e-7 * np.linalg.norm(ref[r] * hs)
    ctx.set_fmm(4.0)                                    # nothing is held any more: all requests are granted
    ctx.apply(np.ones((1, n, 2 * p + 1), dtype=complex))
    ctx.close()


def test_batch_takes_optional_memory_back(L):
    import torch
    p = 8
    ctx, _, _, hs = context(L, 200, p)
    lays = [inputs.layout(k, -inputs.widened_half_width(k), inputs.widened_half_width(k), k) for k in (200, 120, 30)]
    ctx.set_layouts(lays)
    n = ctx.n
    x = torch.from_numpy(inputs.random_coefficients(n, p, 1, 2) / hs).cuda()
    ref, y = torch.zeros_like(x), torch.zeros_like(x)
    ctx.apply_dev(x, ref)                               # captured for the next call with these buffers
    ctx.apply_dev(x, ref)
    beta, _ = ctx.solve([[0.0, 1.0]], tol=1e-10, maxiter=600)
    torch.cuda.synchronize()
    limits(ctx, required=0)
    beta2, _ = ctx.solve([[0.0, 1.0]], tol=1e-10, maxiter=1200)      # a larger basis than before
    assert np.linalg.norm(beta2 * hs - beta * hs) <= 1e-7 * np.linalg.norm(beta * hs)
    ctx.apply_dev(x, ref.clone())
    ctx.apply_dev(x, y)
    first = y.clone()
    ctx.apply_dev(x, y)
    torch.cuda.synchronize()
    for v in (first, y):
        assert rel(v[0].cpu().numpy(), ref[0].cpu().numpy(), hs) <= TOL
    ctx.close()


def test_captured_application_outlives_a_change_to_boxes(L):
    import torch
    n, p = 300, 8
    ctx, c, _, hs = context(L, n, p)
    ctx.set_particles(c)
    x = torch.from_numpy(inputs.random_coefficients(n, p, 1, 2) / hs).cuda()
    y, ref = torch.zeros_like(x), torch.zeros_like(x)
    ctx.apply_dev(x, ref)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.apply_dev(x, y)
    ctx.set_fmm(4.0)
    other = [torch.full((1 << 20,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(8)]
    graph.replay()
    torch.cuda.synchronize()
    assert rel(y[0].cpu().numpy(), ref[0].cpu().numpy(), hs) <= TOL
    del graph, other
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_capture_allocates_nothing(L, precision):
    """A capture that begins before the digit products have run on this layout: after another layout of the
    same size, and after applications that had no need of them."""
    import torch
    n, p = 300, 8
    ctx, c, _, hs = context(L, n, p, precision)
    h = inputs.widened_half_width(n)
    x = torch.from_numpy(inputs.random_coefficients(n, p, 1, 2) / hs).cuda()
    y, ref = torch.zeros_like(x), torch.zeros_like(x)
    for warm in (0, L.APPLY_NO_TRANSLATION):
        ctx.set_particles(inputs.layout(n, -h, h, 77))
        if warm:
            ctx.close()
            ctx, _, _, _ = context(L, n, p, precision)
            ctx.set_particles(c)
        ctx.apply_dev(x, y, warm)
        if not warm:
            ctx.set_particles(c)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ctx.apply_dev(x, y)
        y.zero_()
        graph.replay()
        torch.cuda.synchronize()
        ctx.apply_dev(x, ref)
        torch.cuda.synchronize()
        assert rel(y[0].cpu().numpy(), ref[0].cpu().numpy(), hs) <= TOL
        del graph
    ctx.close()
