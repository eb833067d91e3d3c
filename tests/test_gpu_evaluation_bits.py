"""The evaluation's two launch shapes (parts on warps of their own up to 672 scenarios, one thread per
scenario and stage above) give the same values and partials bit for bit, so that a problem's results
do not depend on the batch that it runs in."""
import numpy as np
import pytest

import absorber_inputs as ai
from test_gpu_parity import B, P, _iterate, dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 672])
def test_values_do_not_depend_on_the_launch_shape(B, n):  # noqa: F811
    import torch
    S = 700
    F, (Z, d, lam) = _iterate(S, 5)
    at = np.arange(S - n, S)                # the same scenarios, at other places of their blocks
    out = []
    for idx in (np.arange(S), at):
        prob = B.Problem(P, F[:, idx])
        x, lm = dev(prob.to_soa(Z[idx], d)), dev(prob.to_soa(lam[idx]))
        new = lambda k: torch.zeros(k * prob.ld, dtype=torch.float64, device="cuda")  # noqa: E731
        for want in ("c", "j", "h", "cj", "cjh"):
            v = {k: new(m) if k in want else None
                 for k, m in (("c", 220), ("j", prob.sizes.nnzJ_scen), ("h", prob.sizes.nnzH_scen))}
            prob.eval_grad_jac_hess(x, lm, 1.0, c=v["c"], jac=v["j"], hess=v["h"])
            out.append([None if t is None else t.view(-1, prob.ld)[:, :len(idx)][:, -n:].clone() for t in v.values()])
    for whole, part in zip(out[:5], out[5:]):
        for a, b in zip(whole, part):
            assert (a is None and b is None) or torch.equal(a, b)
    # nor on the set of outputs that is asked for
    for k in range(3):
        same = [o[k] for o in out[:5] if o[k] is not None]
        assert all(torch.equal(same[0], v) for v in same)


def test_a_problem_alone_and_in_a_batch(B):  # noqa: F811
    # 60 scenarios alone, and beside 650 others of another problem (the partials steer every step)
    import torch
    feeds = [ai.make_feeds(60, 5), ai.make_feeds(650, 6)]
    o = B.default_options(autotune=0)
    alone = B.Problem(P, feeds[0])
    x = torch.zeros(alone.n_primal, dtype=torch.float64, device="cuda")
    r = alone.ipm_solve(o, x_out=x)
    both = B.Batch(P, feeds)
    xb = torch.zeros(both.n_primal, dtype=torch.float64, device="cuda")
    rb = both.ipm_solve(o, x_out=xb)
    assert r.status == 0 and [q.status for q in rb] == [0, 0]
    assert (r.iters, r.E0, r.d) == (rb[0].iters, rb[0].E0, rb[0].d)
    a, b = x[:220 * alone.ld].view(220, alone.ld)[:, :60], xb[:220 * both.ld].view(220, both.ld)[:, :60]
    assert torch.equal(a, b) and x[220 * alone.ld] == xb[220 * both.ld]
