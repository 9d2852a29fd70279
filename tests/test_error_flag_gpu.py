"""A kernel whose bounded wait runs out sets the context's error flag and leaves its sum incomplete.
Every call that returns results of such kernels reads the flag, in FP64 as in mixed precision: it
fails with LSMS_ERR_CUDA, and the next call starts with a clear flag.  The flag is set from the host
here, as the kernels would leave it."""
import ctypes

import numpy as np
import pytest

from paper_1407_3868_gb300 import inputs

pytestmark = pytest.mark.gpu

CUDA = -6


@pytest.fixture(scope="module")
def L():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1407_3868_gb300 import lsms
    return lsms


def raise_flag(ctx, code=21):
    flag = ctx.lib._Z11tc_err_flagP8lsms_ctx          # the library's own accessor
    flag.restype = ctypes.c_void_p
    p = flag(ctx.h)
    assert p
    v = ctypes.c_int(code)
    assert ctypes.CDLL("libcuda.so.1").cuMemcpyHtoD_v2(ctypes.c_ulonglong(p), ctypes.byref(v), ctypes.c_size_t(4)) == 0


@pytest.mark.parametrize("precision", [0, 1])
def test_every_step_reports_the_flag(L, precision):
    n, p = 320, 8
    h = inputs.widened_half_width(n)
    m = inputs.MEDIUM
    ctx = L.Context(m["k1"], m["k2"], m["k3"], m["d"], m["kp"], m["radius"], p, 256, b=inputs.contour_b(2 * h),
                    t_max=141.0, panel_order=16, precision=precision)
    ctx.set_particles(inputs.layout(n, -h, h, 4))
    x = inputs.random_coefficients(n, p, 1, 3)
    sig = np.ones(ctx.ns, dtype=complex)
    src, tgt = [[0.0, 1.0]], [[0.5, 1.0]]
    ctx.solve(src, tol=1e-8, maxiter=400)
    calls = {
        "apply": lambda: ctx.apply(x, L.APPLY_MIXED if precision else 0),
        "translate": lambda: ctx.translate(x, precision=precision),
        "aggregate": lambda: ctx.aggregate(x, precision=precision),
        "disaggregate": lambda: ctx.disaggregate(sig, sig, precision=precision),
        "incident": lambda: ctx.incident(src),
        "eval_field": lambda: ctx.eval_field(tgt, 0, L.FIELD_SCATTERED),
        "solve": lambda: ctx.solve(src, tol=1e-8, maxiter=400),
    }
    for name, call in calls.items():
        raise_flag(ctx)
        with pytest.raises(L.LsmsError) as e:
            call()
        assert e.value.code == CUDA and "21" in str(e.value), name
        call()
    ctx.close()
