"""GPU parity of the FP64 contour contractions against the oracle, through the C ABI, on both sides of
the table size from which they run on the tensor cores (1.5e5 complex elements) and around their
tiles: row tiles of 128 (full, one row), K ranges of 16 (a remainder of one), a partial last drain,
several right-hand sides, the three column paddings.

Tolerance: the repository's 1e-10 for single FP64 steps (phases lambda x up to 1e4 carry 1e-12)."""
import numpy as np
import pytest

from oracle import lsms_oracle as O
from paper_1407_3868_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1407_3868_gb300 import lsms
    return lsms


@pytest.mark.parametrize("n,p,n_nodes,nrhs", [(1, 0, 256, 1), (16, 10, 256, 1), (73, 12, 1024, 1), (74, 12, 1024, 2),
                                              (129, 7, 600, 1), (257, 10, 512, 3), (640, 15, 256, 1), (1000, 3, 384, 1)])
def test_aggregate_and_disaggregate(L, n, p, n_nodes, nrhs):
    m = inputs.MEDIUM
    h = max(2.0, inputs.widened_half_width(n))
    c = inputs.layout(n, -h, h, 40 + n)
    t_max = 60.0 if p <= 3 else 141.0
    ctx = L.Context(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"], p, n_nodes, b=inputs.contour_b(2 * h),
                    t_max=t_max, panel_order=16)
    ctx.set_particles(c)
    lam, wt = ctx.contour()
    pr = O.Problem(O.Medium(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"]), p, c, lam, wt)
    hs = O.order_scale(p, m["k2"], m["radius"])
    x = inputs.random_coefficients(n, p, nrhs, seed=n) / hs
    pp, qm = ctx.aggregate(x)
    a = None
    for r in range(nrhs):
        po, qo = pr.aggregate(x[r])
        assert np.linalg.norm(pp[r] - po) <= TOL * np.linalg.norm(po)
        assert np.linalg.norm(qm[r] - qo) <= TOL * np.linalg.norm(qo)
    sp, sm = ctx.reflect(pp, qm)
    a = ctx.disaggregate(sp, sm)
    for r in range(nrhs):
        ref = pr.disaggregate(sp[r], sm[r])
        assert np.linalg.norm((a[r] - ref) / hs) <= TOL * np.linalg.norm(ref / hs)
    ctx.close()


def test_non_finite_order_stays_in_its_column(L):
    """A NaN in one order of one disc reaches every row of that order alone (as a sum would), in that
    right-hand side alone; zero columns stay zero."""
    import torch
    n, p = 300, 8
    h = inputs.widened_half_width(n)
    m = inputs.MEDIUM
    ctx = L.Context(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"], p, 512, b=inputs.contour_b(2 * h),
                    t_max=141.0, panel_order=16)
    ctx.set_particles(inputs.layout(n, -h, h, 9))
    x = torch.zeros((2, n, 2 * p + 1), dtype=torch.complex128, device="cuda")
    x[1, :, p] = 1.0
    x[0, 5, 3] = complex(float("nan"), 0.0)
    y = torch.zeros_like(x)
    ctx.apply_dev(x, y, L.APPLY_ALPHA | L.APPLY_NO_TRANSLATION)
    torch.cuda.synchronize()
    assert torch.isnan(y[0].real).all() and torch.isfinite(torch.view_as_real(y[1])).all()
    y0 = torch.zeros_like(x)
    ctx.apply_dev(torch.zeros_like(x), y0, L.APPLY_ALPHA | L.APPLY_NO_TRANSLATION)
    torch.cuda.synchronize()
    assert torch.all(y0 == 0)
    ctx.close()
