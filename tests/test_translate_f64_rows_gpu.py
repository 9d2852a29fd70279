"""The FP64 translation keeps every row to its own size when the discs' coefficients are uneven: one
disc larger than all others (its own row does not contain it), two of one size, all in one order, the
same size in every order; below and above the disc count from which even right-hand sides take six
digit levels; through row ranges with and without the large disc.  Against the oracle's pair sums, row by row.

Tolerance: 1e-11 as for the other rows of this translation (phases: 4 * 1.1e-16 * k2 rho, k2 rho <= 5.1e3,
2e-12; operands of 48 bits against |H| >= 0.011: 1e-12).  The large disc's own row is a plain FP64 sum over
CUDA's J and Y, which are good to 5e-12 absolute: 5e-12 / 0.011, 5e-10."""
import numpy as np
import pytest

from oracle import lsms_oracle as O
from paper_1407_3868_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL, TOL_OWN = 1e-11, 5e-10


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1407_3868_gb300 import lsms
    return lsms


def setup(L, n, p):
    m = inputs.MEDIUM
    h = inputs.widened_half_width(n)
    c = inputs.layout(n, -h, h, 60 + n)
    ctx = L.Context(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"], p, 256, b=inputs.contour_b(2 * h),
                    t_max=141.0, panel_order=16)
    ctx.set_particles(c)
    return ctx, c, O.order_scale(p, m["k2"], m["radius"])


def row_errors(a, ref, hs):
    return [np.linalg.norm((a - ref) * w, axis=1) / np.linalg.norm(ref * w, axis=1) for w in (1.0, 1.0 / hs)]


@pytest.mark.parametrize("n,p", [(300, 12), (1100, 9)])
def test_uneven_coefficients(L, n, p):
    ctx, c, hs = setup(L, n, p)
    big, other = n // 3, n - 7
    x = inputs.random_coefficients(n, p, 8, seed=n)
    x[:7] /= hs
    for r, f in enumerate((15.0, 40.0, 1e4, 1e8, 1e14)):       # either side of the 16 that makes a disc dominant
        x[r, big] *= f
    x[5, [big, other]] *= 1e8
    x[6, :, np.arange(2 * p + 1) != p] = 0.0                   # order 0 alone; x[7]: the same size in every order
    a = ctx.translate(x)
    rows = sorted({0, 1, big, other, n // 2, 128, n - 1} | set(np.argsort(np.abs(c[:, 0] - c[big, 0]))[:4].tolist()))
    for r in range(len(x)):
        ref = O.translate(c, x[r], inputs.MEDIUM["k2"], p, rows)
        tol = np.array([TOL_OWN if l == big and r < 5 else TOL for l in rows])
        for e in row_errors(a[r][rows], ref, hs):
            assert np.all(e <= tol), (r, dict(zip(rows, e)))
    ctx.close()


def test_row_ranges_with_and_without_the_large_disc(L):
    import torch
    n, p = 300, 8
    ctx, c, hs = setup(L, n, p)
    big = 130
    x = inputs.random_coefficients(n, p, 2, seed=5) / hs
    x[1, big] *= 1e9
    xd = torch.from_numpy(x).cuda()
    ref = [O.translate(c, x[r], inputs.MEDIUM["k2"], p) for r in range(2)]
    for row0, row1 in ((0, 130), (130, 131), (100, 300), (131, 300)):
        y = torch.zeros((2, row1 - row0, 2 * p + 1), dtype=torch.complex128, device="cuda")
        ctx.apply_rows_dev(xd, y, row0, row1, L.APPLY_ALPHA | L.APPLY_NO_REFLECTION)
        torch.cuda.synchronize()
        for r in range(2):
            tol = np.array([TOL_OWN if l == big and r else TOL for l in range(row0, row1)])
            for e in row_errors(y[r].cpu().numpy(), ref[r][row0:row1], hs):
                assert np.all(e <= tol), (row0, r, e.max())
    ctx.close()
