"""Box widths that are refused (more than 131072 boxes) leave a context that translates over all pairs,
against the oracle's pair sums: refused by lsms_set_fmm after a width that was accepted, and by
lsms_set_particles for a layout too long for the width set before.  Layouts with digit products (few
near pairs) and with all pairs stored (mostly near pairs).

Tolerance: 1e-11, as for the other FP64 translations (k2 rho up to 3.5e4 at 4 * 1.1e-16 each is 1.6e-11
on the farthest pairs alone, whose |H| is 40 times below that of the near ones)."""
import numpy as np
import pytest

from oracle import lsms_oracle as O
from paper_1407_3868_gb300 import inputs

pytestmark = pytest.mark.gpu

ARG = -1
TOL = 1e-11
P_ORDER, K2, R, D = 5, 0.5, 0.2, 1.0


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1407_3868_gb300 import lsms
    return lsms


def context(L):
    return L.Context(0.4, K2, 0.45, D, 0.45, R, P_ORDER, 128, b=0.01, t_max=60.0, panel_order=16)


def layout(half_width):
    c = inputs.layout(118, -half_width, half_width, 3, radius=R, d=D)
    return np.concatenate([c, [[-70000.0, -0.5], [70000.0, -0.4]]])


def check(ctx, c):
    hs = O.order_scale(P_ORDER, K2, R)
    x = inputs.random_coefficients(len(c), P_ORDER, 1, 8) / hs
    a = ctx.translate(x)[0]
    ref = O.translate(c, x[0], K2, P_ORDER)
    assert np.linalg.norm((a - ref) / hs) <= TOL * np.linalg.norm(ref / hs)


@pytest.mark.parametrize("half_width", [400.0, 40.0])
def test_narrower_boxes_refused(L, half_width):
    c = layout(half_width)
    with context(L) as ctx:
        ctx.set_particles(c)
        check(ctx, c)
        ctx.set_fmm(500.0)
        with pytest.raises(L.LsmsError) as e:
            ctx.set_fmm(1.0)
        assert e.value.code == ARG and "131072 boxes" in str(e.value)
        assert ctx.fmm_info()[0] == 0
        check(ctx, c)


@pytest.mark.parametrize("half_width", [400.0, 40.0])
def test_layout_too_long_for_the_boxes(L, half_width):
    c = layout(half_width)
    with context(L) as ctx:
        ctx.set_fmm(1.0)
        ctx.set_particles(c[:118])
        with pytest.raises(L.LsmsError) as e:
            ctx.set_particles(c)
        assert e.value.code == ARG and "131072 boxes" in str(e.value)
        assert ctx.lib.lsms_num_particles(ctx.h) == len(c)
        ctx.n = len(c)
        check(ctx, c)
        ctx.set_fmm(0.0)
        check(ctx, c)
