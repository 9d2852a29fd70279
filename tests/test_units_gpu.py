"""The FP64 translation does not depend on the unit of length: the same layout and medium with lengths scaled
by a power of two near 1e-25 and 1e25 gives the same coefficients (which have no unit).  Short layouts
and layouts with digit products.

Tolerance: 1e-11 in the scaled norm, as for the FP64 translation against the oracle (powers of two change
no rounding of the phases)."""
import numpy as np
import pytest

from oracle import lsms_oracle as O
from paper_1407_3868_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1407_3868_gb300 import lsms
    return lsms


@pytest.mark.parametrize("n", [40, 200])
def test_unit_of_length(L, n):
    p, m = 8, inputs.MEDIUM
    h = inputs.widened_half_width(n)
    c = inputs.layout(n, -h, h, 12)
    hs = O.order_scale(p, m["k2"], m["radius"])
    x = inputs.random_coefficients(n, p, 1, 3) / hs
    out = []
    for u in (1.0, 2.0 ** -83, 2.0 ** 83):
        with L.Context(m["k1"] / u, m["k2"] / u, m["k3"] / u, m["d"] * u, m["kp"] / u, m["radius"] * u, p, 384,
                       b=inputs.contour_b(2 * h) / u, t_max=141.0 / u, panel_order=16) as ctx:
            ctx.set_particles(c * u)
            out.append(ctx.translate(x)[0])
    for t in out[1:]:
        assert np.linalg.norm((t - out[0]) / hs) <= 1e-11 * np.linalg.norm(out[0] / hs)
