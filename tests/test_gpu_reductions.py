"""The per-problem reductions (reduce_kernel) around one chunk of 256 (stage, scenario) elements (25
and 26 scenarios) and around the 256 chunks whose results a warp combines in one round (6553 and
6554 scenarios): the sums of a Newton direction (the Schur complement of the design, its residual
norms) through the checks of test_gpu_condensed, and a NaN among them."""
import math

import pytest

import test_gpu_condensed as cond
from test_gpu_condensed import B  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [25, 26, 6553, 6554])
def test_sums_and_maxima(B, S):  # noqa: F811
    import torch
    cond.test_direction_solves_the_system(B, S, 0)
    prob, x, jac, hes, sig, rx, rc = cond._system(B, S)
    prob.kkt_factor(x, jac, hes, sig, delta_w=1e-3)
    sx, sc = torch.zeros_like(rx), torch.zeros_like(rc)
    for at in (0, S - 1):
        bad = rc.clone()
        bad[219 * prob.ld + at] = float("nan")
        prob.kkt_solve(rx, bad, sx, sc, max_refine=0)
        assert torch.isnan(sx[-1])   # the sum behind the design's step
    info = prob.kkt_solve(rx, rc, sx, sc, max_refine=1)   # the next solve is not affected
    assert math.isfinite(info.residual)
