"""The tensor-core FP32 factor (ABS_PREC_FP32_TC, options.factor_kernel = 1) is the only factorization
of its systems: condensed factors besides it belong to the escalations and second-order corrections of
a solve."""
import pytest

import absorber_inputs as ai
import test_gpu_condensed as cond
from test_gpu_condensed import B  # noqa: F401

pytestmark = pytest.mark.gpu
P = ai.PARAMS


def test_one_factorization_per_iteration(B):  # noqa: F811
    F = ai.make_feeds(60, 5)
    res = []
    for k in (0, 1):
        prob = B.Problem(P, F)
        # six iterations from the inlet-copy start (no FP64 solve for a start), no corrections
        res.append(prob.ipm_solve(B.default_options(precision=1, max_refine=8, factor_kernel=k, soc_max=0, init=1,
                                                    max_iter=6, graphs=0, autotune=0)))
        assert res[-1].iters == 6 and res[-1].fp64_fallbacks == 0 and res[-1].base_iters == 0
    kf = B.KINDS.index("factor")
    # condensed factors take two launches a factorization, the tensor-core factor one
    two, one = (r.kind_launches[kf] for r in res)
    assert 2 * one == two


def test_factor_holds_its_own_storage_only(B):  # noqa: F811
    # 22 x 22 inverses and 22 x 11 blocks of ten stages in FP32, and the row orders: 29.5 KB a
    # scenario; the condensed factors would be another 10 KB
    import torch
    S = 20000
    prob, x, jac, hes, sig, rx, rc = cond._system(B, S)
    prob.kkt_factor(x, jac, hes, sig, precision=0)        # the handle's vectors are there
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    prob.kkt_factor(x, jac, hes, sig, precision=3)
    used = free - torch.cuda.mem_get_info()[0]
    own = S * (10 * 4 * (22 * 22 + 22 * 11) + 10 * 44)
    assert used <= own + (16 << 20), (used, own)


@pytest.mark.parametrize("prec", [1, 3])
@pytest.mark.parametrize("S", [5, 300])
def test_directions_before_and_after_a_solve(B, S, prec):  # noqa: F811
    # a solve with the other FP32 factor, or in FP64, leaves kkt_factor and kkt_solve what they were
    import torch
    prob, x, jac, hes, sig, rx, rc = cond._system(B, S)
    ref = None
    for opt in (None, dict(precision=0), dict(precision=1, factor_kernel=1, max_refine=8),
                dict(precision=1, factor_kernel=0, max_refine=8)):
        if opt is not None:
            assert prob.ipm_solve(B.default_options(autotune=0, **opt)).status == 0
        prob.kkt_factor(x, jac, hes, sig, delta_w=1e-3, precision=prec)
        a, b = torch.zeros_like(rx), torch.zeros_like(rc)
        info = prob.kkt_solve(rx, rc, a, b, max_refine=3)
        if ref is None:
            ref = a, b, info.residual
        assert info.residual == ref[2] and torch.equal(a, ref[0]) and torch.equal(b, ref[1])
