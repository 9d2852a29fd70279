"""GPU parity of the FP64 translation on the tensor cores (layouts from 96 discs on) against the
oracle's pair sums, through the C ABI.

Sizes around its tiles: the first layout that takes it (96; 95 keeps the FP64 pipe), 128-target
tiles with a full, one-row and nearly full last tile, odd source counts (a drain group of one
source), the change from seven to six digit levels at 1024 discs; orders at the edges of the three
column paddings (7, 8, 11, 12, 15) and the smallest.

Tolerance: the phase k2 rho of a pair carries at most about four FP64 roundings, 4 * 1.1e-16 * k2 rho,
with k2 rho <= 5e3 here: 2e-12; five times that, 1e-11, on the sampled rows in the scaled norm.
"""
import numpy as np
import pytest

from oracle import lsms_oracle as O
from paper_1407_3868_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 1e-11


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1407_3868_gb300 import lsms
    return lsms


def context(L, n, p, seed):
    h = inputs.widened_half_width(n)
    m = inputs.MEDIUM
    c = inputs.layout(n, -h, h, seed)
    ctx = L.Context(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"], p, 256, b=inputs.contour_b(2 * h),
                    t_max=141.0, panel_order=16)
    ctx.set_particles(c)
    return ctx, c


def rows_of(n):
    return sorted({0, 1, 127 % n, 128 % n, n // 2, n - 2, n - 1})


@pytest.mark.parametrize("n,p,nrhs", [(95, 10, 1), (96, 0, 1), (96, 7, 2), (127, 8, 1), (128, 11, 1), (129, 12, 3),
                                      (257, 15, 1), (640, 3, 1), (1023, 12, 1), (1024, 14, 1), (1025, 15, 2)])
def test_translation_against_pair_sums(L, n, p, nrhs):
    ctx, c = context(L, n, p, 300 + n)
    hs = O.order_scale(p, inputs.MEDIUM["k2"], inputs.MEDIUM["radius"])
    x = inputs.random_coefficients(n, p, nrhs, seed=n) / hs
    a = ctx.translate(x)
    rows = rows_of(n)
    for r in range(nrhs):
        ref = O.translate(c, x[r], inputs.MEDIUM["k2"], p, rows)
        got = a[r][rows]
        for weight in (1.0 / hs, np.eye(1, 2 * p + 1, p)[0]):       # scaled norm; order 0 alone (far pairs)
            assert np.linalg.norm((got - ref) * weight) <= TOL * np.linalg.norm(ref * weight)
    ctx.close()


@pytest.mark.parametrize("scale", [1e-200, 1.0, 1e200])
def test_scale_and_uneven_columns(L, scale):
    """Right-hand sides scale exactly, a zero one stays zero, and one that lives on a single disc (a
    power-of-two multiple of it) equals its column."""
    n, p = 130, 9
    ctx, c = context(L, n, p, 77)
    hs = O.order_scale(p, inputs.MEDIUM["k2"], inputs.MEDIUM["radius"])
    x = np.zeros((3, n, 2 * p + 1), dtype=complex)
    x[0] = inputs.random_coefficients(n, p, 1, seed=4)[0] / hs
    x[2, 17] = x[0, 17]
    a = ctx.translate(scale * x)
    assert np.all(a[1] == 0)
    rows = [0, 5, 64, 129]
    for r in (0, 2):
        ref = scale * O.translate(c, x[r], inputs.MEDIUM["k2"], p, rows)
        assert np.max(np.abs(a[r][rows] - ref) / hs) <= TOL * np.max(np.abs(ref) / hs)
    assert np.all(a[2, 17] == 0)
    ctx.close()


def test_non_finite_coefficients_reach_every_row(L):
    import torch
    n, p = 200, 10
    ctx, _ = context(L, n, p, 78)
    x = torch.zeros((2, n, 2 * p + 1), dtype=torch.complex128, device="cuda")
    x[0, 3, 4] = complex(float("nan"), 0.0)
    x[1, :, p] = 1.0
    y = torch.zeros_like(x)
    ctx.apply_dev(x, y, L.APPLY_ALPHA | L.APPLY_NO_REFLECTION)
    torch.cuda.synchronize()
    assert torch.isnan(y[0].real).all() and torch.isfinite(torch.view_as_real(y[1])).all()
    ctx.close()
