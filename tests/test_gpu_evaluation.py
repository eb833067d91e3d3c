"""The evaluation's launch shapes (four warps per 32 scenarios and stage up to 672 scenarios, one
thread per scenario and stage above) with every set of outputs, at one scenario, ragged blocks and
both sides of that line, against the oracle's derivatives on sampled scenarios.  Tolerances of the
parity tests: the same closed forms in FP64, 1e-11 of a row's largest entry."""
import numpy as np
import pytest

from oracle import model
from test_gpu_parity import B, P, _iterate, _rowscaled_close, dev, host  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 31, 32, 33, 672, 673, 1217])
def test_values_of_every_output_set(B, S):  # noqa: F811
    import torch
    F, (Z, d, lam) = _iterate(S, S)
    prob = B.Problem(P, F)
    x, lm = dev(prob.to_soa(Z, d)), dev(prob.to_soa(lam))
    jr, jc, hr, hc = prob.pattern()
    idx = np.unique([0, S // 2, max(0, S - 33), S - 1])
    Co, J, Jd, W, Wdd = model.derivatives(P, F[:, idx], Z[idx], d, lam[idx])
    Jo = np.concatenate([J, Jd[:, :, None]], axis=2)[:, jr, jc]
    Wf = np.zeros((len(idx), model.NS + 1, model.NS + 1))
    Wf[:, :model.NS, :model.NS] = W
    Wf[:, model.NS, model.NS] = Wdd
    Ho = Wf[:, hr, hc]
    new = lambda n: torch.full((n * prob.ld,), np.nan, dtype=torch.float64, device="cuda")  # noqa: E731
    for want in ("c", "j", "h", "cj", "cjh", "jh", "ch"):
        c = new(model.NS) if "c" in want else None
        j = new(len(jr)) if "j" in want else None
        h = new(len(hr)) if "h" in want else None
        prob.eval_grad_jac_hess(x, lm, 1.0, c=c, jac=j, hess=h)
        if c is not None:
            _rowscaled_close(prob.values_to_scen(host(c), model.NS)[idx], Co, np.arange(model.NS), 1e-11, floor=1e-12)
        if j is not None:
            _rowscaled_close(prob.values_to_scen(host(j), len(jr))[idx], Jo, jr, 1e-11)
        if h is not None:
            _rowscaled_close(prob.values_to_scen(host(h), len(hr))[idx], Ho, hr, 1e-11)
