"""The FP64 reflected coupling and its densities keep small outputs to their own size: coefficients that
are uneven over the discs and over the orders, checked disc by disc in the unscaled norm (where the
highest orders weigh) and node by node, against the oracle.  Layouts of all depths, of one depth (one
depth class) and of two, and in a layer six times as thick (twice as many classes); nine right-hand sides at once, more than one block of images holds at p = 15.

Tolerance: the repository's 1e-10 for single FP64 steps, here for every disc's row and every node by
itself; the FP64 phases lambda x (up to 1e4) carry about 1e-12 of it.  Where a row's terms cancel (a
thousandfold at most here) those phases alone, the oracle's among them, can pass 1e-10: the row may then be twice as
far off as the same coupling taken in its single steps, whose sums are plain FP64 ones."""
import numpy as np
import pytest

from oracle import lsms_oracle as O
from paper_1407_3868_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 1e-10
TINY = 1e-290            # what underflows on the way (e^{-Re gamma t} in the thick layer) has no digits to compare


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1407_3868_gb300 import lsms
    return lsms


def coefficients(n, p, hs, c):
    x = inputs.random_coefficients(n, p, 9, seed=n + p)
    shallow, deep = int(np.argmax(c[:, 1])), int(np.argmin(c[:, 1]))
    only = lambda v, j: np.where(np.arange(n)[:, None] == j, v, 0.0)  # noqa: E731
    x[0] /= hs                                        # what GMRES sees; x[1]: the same size in every order
    x[2] = only(x[2] / hs, deep)
    x[3] = only(x[3] / hs, shallow)
    x[4] = np.where(np.arange(n)[:, None] == deep, 1e8, 1.0) * x[4] / hs
    x[5] = np.where(np.arange(n)[:, None] == shallow, 1e8, 1.0) * x[5] / hs
    x[6] = 0.0
    x[7] = only(np.where(np.arange(2 * p + 1) == p, x[7], 0.0), deep)
    x[8] = x[8] / hs * np.exp(20.0 * c[:, 1:] / 2.0)  # falling with depth
    return x, deep


@pytest.mark.parametrize("kind,n,p,n_nodes", [("all", 300, 12, 512), ("one", 300, 9, 384), ("two", 200, 7, 512),
                                              ("all", 640, 15, 256), ("thick", 400, 10, 512)])
def test_rows_and_nodes(L, kind, n, p, n_nodes):
    m = dict(inputs.MEDIUM, d=12.0 if kind == "thick" else inputs.MEDIUM["d"])
    h = inputs.widened_half_width(n) if kind in ("all", "thick") else 0.35 * n
    c = inputs.layout(n, -h, h, 11, d=m["d"])
    if kind in ("one", "two"):
        c = np.stack([np.linspace(-h, h, n), np.full(n, -1.0)], axis=1)
        if kind == "two":
            c[::2, 1], c[1::2, 1] = -0.31, -1.69
    ctx = L.Context(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"], p, n_nodes, b=inputs.contour_b(2 * h),
                    t_max=141.0, panel_order=16)
    ctx.set_particles(c)
    lam, wt = ctx.contour()
    pr = O.Problem(O.Medium(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"]), p, c, lam, wt)
    hs = O.order_scale(p, m["k2"], m["radius"])
    x, deep = coefficients(n, p, hs, c)
    a = ctx.apply(x, L.APPLY_ALPHA | L.APPLY_NO_TRANSLATION)
    pp, qm = ctx.aggregate(x)
    assert np.all(a[6] == 0) and np.all(pp[6] == 0)
    steps = ctx.disaggregate(*ctx.reflect(pp, qm))
    for r in range(len(x)):
        if r == 6:
            continue
        ref = pr.reflection(x[r])
        for w in (1.0, 1.0 / hs):
            rows, plain = (np.linalg.norm((v[r] - ref) * w, axis=1) / np.linalg.norm(ref * w, axis=1) for v in (a, steps))
            assert np.all(rows <= np.maximum(TOL, 2 * plain)), (r, rows.max(), plain.max())
        if r in (2, 3, 7):                            # a single disc: no cancellation between discs
            po, qo = pr.aggregate(x[r])
            assert np.all(np.abs(pp[r] - po) <= TOL * np.abs(po) + TINY), r
            assert np.all(np.abs(qm[r] - qo) <= TOL * np.abs(qo) + TINY), r
    # incident coefficients of sources high above the layer and close to it
    for src in ([0.3, 1.0], [-0.4, 0.05]):
        ref = pr.incident_local(np.array(src))
        got = ctx.incident([src])[0]
        for w in (1.0, 1.0 / hs):
            assert np.max(np.linalg.norm((got - ref) * w, axis=1) / np.linalg.norm(ref * w, axis=1)) <= TOL, src
    # one node alone: the deep discs' rows of an evanescent density
    s = np.zeros(len(lam), dtype=complex)
    s[int(np.argmin(np.abs(lam.real - 60.0)))] = 1.0
    d = ctx.disaggregate(s, np.zeros_like(s))[0]
    ref = pr.disaggregate(s, np.zeros_like(s))
    assert np.all(np.abs(d - ref) <= TOL * np.abs(ref) + TINY)
    ctx.close()
