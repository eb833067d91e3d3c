"""A direction written over its own right-hand side (no refinement, which would need it again) is the
one written elsewhere, bit for bit."""
import pytest

import test_gpu_condensed as cond
from test_gpu_condensed import B, P  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1, 3, 4])
@pytest.mark.parametrize("S", [1, 5, 6, 7, 130, 6000])
def test_kkt_solve_in_place(B, S, prec):  # noqa: F811
    import torch
    if prec == 4 and S > 1000:
        pytest.skip("block LDL^T: small sizes")
    prob, x, jac, hes, sig, rx, rc = cond._system(B, S)
    prob.kkt_factor(x, jac, hes, sig, delta_w=1e-3, precision=prec)
    sx, sc = torch.zeros_like(rx), torch.zeros_like(rc)
    go = lambda *v: B.lib().kkt_solve(prob.h, *[t.data_ptr() for t in v], 0, 1e-14, None, None)  # noqa: E731
    assert go(rx, rc, sx, sc) == 0
    ax, ac = rx.clone(), rc.clone()
    assert go(ax, ac, ax, ac) == 0
    torch.cuda.synchronize()
    live = lambda v: v[:220 * prob.ld].view(220, prob.ld)[:, :S]  # noqa: E731
    assert torch.equal(live(sx), live(ax)) and torch.equal(live(sc), live(ac)) and sx[-1] == ax[-1]


@pytest.mark.parametrize("S", [1, 7, 128])
def test_newton_noalloc_in_place(B, S):  # noqa: F811
    import torch
    prob, x, jac, hes, sig, rx, rc = cond._system(B, S)
    sx, sc = torch.zeros_like(rx), torch.zeros_like(rc)
    B.kkt_newton_noalloc(P, S, prob.ld, x, jac, hes, sig, rx, rc, sx, sc, delta_w=1e-3)
    ax, ac = rx.clone(), rc.clone()
    B.kkt_newton_noalloc(P, S, prob.ld, x, jac, hes, sig, ax, ac, ax, ac, delta_w=1e-3)
    live = lambda v: v[:220 * prob.ld].view(220, prob.ld)[:, :S]  # noqa: E731
    assert torch.equal(live(sx), live(ax)) and torch.equal(live(sc), live(ac)) and sx[-1] == ax[-1]
