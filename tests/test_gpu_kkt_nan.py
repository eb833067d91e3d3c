"""A NaN in a KKT solve is not a solved system: kkt_solve reports it as its residual, and as
ABS_ERR_NUMERIC where it was to refine; the next solve is not affected."""
import math

import pytest

import test_gpu_condensed as cond
from test_gpu_condensed import B  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1, 3, 4])
@pytest.mark.parametrize("S", [1, 40])
def test_nan_is_reported(B, S, prec):  # noqa: F811
    import ctypes as C

    import torch
    prob, x, jac, hes, sig, rx, rc = cond._system(B, S)
    prob.kkt_factor(x, jac, hes, sig, delta_w=1e-3, precision=prec)
    sx, sc = torch.zeros_like(rx), torch.zeros_like(rc)
    before = prob.kkt_solve(rx, rc, sx, sc, max_refine=8)
    good = sx.clone(), sc.clone()
    bad_x, bad_c, bad_d = rx.clone(), rc.clone(), rx.clone()
    bad_x[5 * prob.ld + S - 1] = math.nan
    bad_c[219 * prob.ld] = math.nan
    bad_d[-1] = math.nan
    for a, b in ((bad_x, rc), (rx, bad_c), (bad_d, rc)):
        assert math.isnan(prob.kkt_solve(a, b, sx, sc, max_refine=0).residual)
        with pytest.raises(B.AbsorberError) as e:
            prob.kkt_solve(a, b, sx, sc, max_refine=2)
        assert e.value.status == -7
        info = B.AbsSolveInfo()
        st = B.lib().kkt_solve(prob.h, a.data_ptr(), b.data_ptr(), sx.data_ptr(), sc.data_ptr(), 2, 1e-14,
                               C.byref(info), None)
        assert st == -7 and math.isnan(info.residual) and info.refine_steps == 0
    sx.zero_(), sc.zero_()
    after = prob.kkt_solve(rx, rc, sx, sc, max_refine=8)
    assert (after.residual, after.refine_steps) == (before.residual, before.refine_steps)
    assert torch.isfinite(sx[-1]) and torch.equal(sx, good[0]) and torch.equal(sc, good[1])
