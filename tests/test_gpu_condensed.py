"""The condensed factors (kernels_cond.cuh) at the edges of their launch shapes: one scenario,
blocks of 4, 6, 8 and 32 scenarios full and ragged, both sides of the size at which the FP64 chain
changes its blocks (4256 scenarios), and singular blocks.

The direction is put back into the dense KKT system of sampled scenarios.  Tolerance: the
elimination's multipliers are at most 7 and its cores have condition below 1e5, so the backward
error of an unrefined FP64 direction stays within a few hundred unit roundoffs of |K| |sol| +
|rhs| summed over a row of at most 45 entries: 1e-12 of that; FP32 factors reach the same after
refinement."""
import numpy as np
import pytest

import absorber_inputs as ai
from oracle import model

pytestmark = pytest.mark.gpu
P = ai.PARAMS


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_15420_gb300 import build
    build.build()
    from paper_2607_15420_gb300 import binding
    binding.lib()
    return binding


def _system(B, S):
    import torch
    F = ai.make_feeds(S, 21)
    rng = np.random.default_rng(S)
    Z, d = model.initial_point(P, F)
    Z = (np.abs(Z) + 0.02) * rng.uniform(0.8, 1.25, Z.shape)
    prob = B.Problem(P, F)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    x, lam = dev(prob.to_soa(Z, d)), dev(prob.to_soa(0.1 * rng.standard_normal(Z.shape)))
    sig = dev(prob.to_soa(rng.uniform(0.5, 2.0, Z.shape), 1.0))
    rx, rc = dev(prob.to_soa(rng.standard_normal(Z.shape), float(S))), dev(prob.to_soa(rng.standard_normal(Z.shape)))
    jac = torch.zeros(prob.sizes.nnzJ_scen * prob.ld, dtype=torch.float64, device="cuda")
    hes = torch.zeros(prob.sizes.nnzH_scen * prob.ld, dtype=torch.float64, device="cuda")
    prob.eval_grad_jac_hess(x, lam, 1.0, jac=jac, hess=hes)
    return prob, x, jac, hes, sig, rx, rc


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("S", [1, 3, 4, 5, 6, 7, 32, 33, 2437, 4255, 4256, 4867])
def test_direction_solves_the_system(B, S, prec):
    import torch
    dw = 1e-3
    prob, x, jac, hes, sig, rx, rc = _system(B, S)
    inert = prob.kkt_factor(x, jac, hes, sig, delta_w=dw, precision=prec)
    assert inert.n_singular == 0 and inert.n_pos + inert.n_neg == 440 * S + 1
    sx, sc = torch.zeros_like(rx), torch.zeros_like(rc)
    prob.kkt_solve(rx, rc, sx, sc, max_refine=(0 if prec == 0 else 8), refine_tol=1e-15)
    h = lambda t: t.cpu().numpy()  # noqa: E731
    dz, dd = prob.from_soa(h(sx))
    dl, _ = prob.from_soa(h(sc))
    rz, rd = prob.from_soa(h(rx))
    rr, _ = prob.from_soa(h(rc))
    sg, sgd = prob.from_soa(h(sig))
    jr, jc, hr, hc = prob.pattern()
    J = prob.values_to_scen(h(jac), len(jr))
    H = prob.values_to_scen(h(hes), len(hr))
    row_d = rd - (H[:, -1].sum() + sgd + dw) * dd
    mag_d = abs(rd)
    for s in range(S):
        on_d = jc == 220
        t = J[s, on_d] * dl[s, jr[on_d]]
        row_d -= t.sum()
        mag_d += np.abs(t).sum()
    assert abs(row_d) <= 1e-12 * mag_d
    for s in sorted({0, 1, S // 2, S - 2, S - 1} & set(range(S))):
        Jf = np.zeros((220, 221))
        Jf[jr, jc] = J[s]
        W = np.zeros((220, 220))
        W[hr[:-1], hc[:-1]] = H[s, :-1]
        W[hc[:-1], hr[:-1]] = H[s, :-1]
        W[np.arange(220), np.arange(220)] += sg[s] + dw
        z = rz[s] - W @ dz[s] - Jf[:, :220].T @ dl[s]
        c = rr[s] - Jf[:, :220] @ dz[s] - Jf[:, 220] * dd
        zm = np.abs(rz[s]) + np.abs(W) @ np.abs(dz[s]) + np.abs(Jf[:, :220]).T @ np.abs(dl[s])
        cm = np.abs(rr[s]) + np.abs(Jf[:, :220]) @ np.abs(dz[s]) + np.abs(Jf[:, 220] * dd)
        assert np.max(np.abs(z)) <= 1e-12 * np.max(zm), s
        assert np.max(np.abs(c)) <= 1e-12 * np.max(cm), s


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("S,bad", [(6, 5), (4900, 31)])
def test_singular_scenario_is_reported(B, S, bad, prec):
    # every Jacobian value of one scenario zeroed: that scenario and no other is singular
    prob, x, jac, hes, sig, _, _ = _system(B, S)
    jac.view(-1, prob.ld)[:, bad] = 0.0
    inert = prob.kkt_factor(x, jac, hes, sig, precision=prec, check=False)
    assert inert.n_singular == 1
    st = prob.scenario_status()
    assert st[bad] == -7 and np.count_nonzero(st) == 1
