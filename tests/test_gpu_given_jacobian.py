"""kkt_factor, kkt_solve and kkt_newton_noalloc with Jacobian values that are not the evaluation's: rows
scaled, an extent's or the slack's coefficient changed, a stream's entry changed in one of the two
stages that it joins, a stage whose H2O pivot cancels, values that differ by rounding.  The condensed
factors assume the first of these and must not be used for them.

The direction is put back into the dense KKT system of every edited scenario, as in
test_gpu_condensed, with its tolerance."""
import numpy as np
import pytest

import test_gpu_condensed as cond
from test_gpu_condensed import B, P  # noqa: F401

pytestmark = pytest.mark.gpu
NV, LV, LT, LE, LS, R_E, R_H, R_SX, R_RX = 22, 14, 15, 16, 21, 20, 21, 18, 13


def _at(jr, jc, row, col):
    i = np.flatnonzero((jr == row) & (jc == col))
    assert i.size == 1
    return int(i[0])


def _edit(kind, J, jr, jc, rng):
    """J [nnz, S] (host), changed in place; the scenarios that were."""
    S = J.shape[1]
    s, n = S - 1, 4
    at = lambda m, row, k, col: _at(jr, jc, NV * m + row, NV * k + col)  # noqa: E731
    if kind == "rows":           # every row but the hydraulic ones (whose design entries come from x)
        scale = rng.uniform(0.3, 3.0, 10 * NV)
        scale[R_H::NV] = 1.0
        J *= scale[jr][:, None]
        return range(S)
    if kind == "extent":
        J[at(n, 4, n, LE + 3), s] *= 1.5
    elif kind == "slack":
        J[at(n, R_H, n, LS), s] = 2.0
    elif kind == "liquid":       # stage n's MEA in the row of the stage below
        J[at(n - 1, 0, n, 0), s] *= 1.01
    elif kind == "vapour":       # stage n's N2 in the row of the stage above
        J[at(n + 1, 9, n, 9 + 2), s] *= 1.01
    elif kind == "flow":
        J[at(n + 1, R_E, n, LV), s] *= 0.99
    elif kind == "heat":         # the two shares of dT in the energy rows
        J[at(n + 1, R_E, n, LT), s] *= 1.01
    elif kind == "pivot":        # sum x: the entry of H2O against those of the species that follow it
        e = lambda row, col: J[at(n, row, n, col), s]  # noqa: E731
        x4 = -e(R_RX + 3, 8) / e(R_RX + 3, 4)
        x5 = -e(R_RX + 2, 8) / e(R_RX + 2, 5)
        x6 = -e(R_RX + 1, 4) / e(R_RX + 1, 6) * x4
        x7 = -(e(R_RX + 4, 4) * x4 + e(R_RX + 4, 8)) / e(R_RX + 4, 7)
        J[at(n, R_SX, n, 8), s] = -(e(R_SX, 4) * x4 + e(R_SX, 5) * x5 + e(R_SX, 6) * x6 + e(R_SX, 7) * x7) * (1 + 1e-13)
    else:                        # rounding
        J *= 1.0 + rng.uniform(-4.0, 4.0, J.shape) * 2.0 ** -53
        return range(min(S, 4))
    return sorted({0, s})


def _residual(prob, J, H, sg, rz, rr, dz, dl, dd, dw, jr, jc, hr, hc, s):
    Jf = np.zeros((220, 221))
    Jf[jr, jc] = J[:, s]
    W = np.zeros((220, 220))
    W[hr[:-1], hc[:-1]] = H[s, :-1]
    W[hc[:-1], hr[:-1]] = H[s, :-1]
    W[np.arange(220), np.arange(220)] += sg[s] + dw
    z = rz[s] - W @ dz[s] - Jf[:, :220].T @ dl[s]
    c = rr[s] - Jf[:, :220] @ dz[s] - Jf[:, 220] * dd
    zm = np.abs(rz[s]) + np.abs(W) @ np.abs(dz[s]) + np.abs(Jf[:, :220]).T @ np.abs(dl[s])
    cm = np.abs(rr[s]) + np.abs(Jf[:, :220]) @ np.abs(dz[s]) + np.abs(Jf[:, 220] * dd)
    return np.max(np.abs(z)) / np.max(zm), np.max(np.abs(c)) / np.max(cm)


KINDS = ("rows", "extent", "slack", "liquid", "vapour", "flow", "heat", "pivot", "rounding")


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("S,prec", [(1, 0), (33, 0), (33, 1), (700, 1)])
def test_direction_solves_the_given_system(B, kind, S, prec):  # noqa: F811
    import torch
    dw = 1e-3
    prob, x, jac, hes, sig, rx, rc = cond._system(B, S)
    jr, jc, hr, hc = prob.pattern()
    Jd = jac.view(len(jr), prob.ld)
    J = Jd[:, :S].cpu().numpy().copy()
    seen = _edit(kind, J, jr, jc, np.random.default_rng(7))
    Jd[:, :S] = torch.from_numpy(J).cuda()
    inert = prob.kkt_factor(x, jac, hes, sig, delta_w=dw, precision=prec)
    assert inert.n_singular == 0 and inert.n_pos + inert.n_neg == 440 * S + 1
    sx, sc = torch.zeros_like(rx), torch.zeros_like(rc)
    prob.kkt_solve(rx, rc, sx, sc, max_refine=(0 if prec == 0 else 8), refine_tol=1e-15)
    h = lambda t: t.cpu().numpy()  # noqa: E731
    dz, dd = prob.from_soa(h(sx))
    dl, _ = prob.from_soa(h(sc))
    args = prob.values_to_scen(h(hes), len(hr)), prob.from_soa(h(sig))[0], prob.from_soa(h(rx))[0], prob.from_soa(h(rc))[0]
    for s in list(seen)[:8]:
        z, c = _residual(prob, J, *args, dz, dl, dd, dw, jr, jc, hr, hc, s)
        assert z <= 1e-12 and c <= 1e-12, s


@pytest.mark.parametrize("kind", KINDS)
def test_direction_without_allocation(B, kind):  # noqa: F811
    import torch
    S = 40
    prob, x, jac, hes, sig, rx, rc = cond._system(B, S)
    jr, jc, hr, hc = prob.pattern()
    Jd = jac.view(len(jr), prob.ld)
    J = Jd[:, :S].cpu().numpy().copy()
    seen = _edit(kind, J, jr, jc, np.random.default_rng(7))
    own = torch.zeros_like(rx), torch.zeros_like(rc)
    B.kkt_newton_noalloc(P, S, prob.ld, x, jac, hes, sig, rx, rc, *own, delta_w=1e-3)
    given = jac.clone()
    given.view(len(jr), prob.ld)[:, :S] = torch.from_numpy(J).cuda()
    sx, sc = torch.full_like(rx, np.nan), torch.full_like(rc, np.nan)
    sd = B.kkt_newton_noalloc(P, S, prob.ld, x, given, hes, sig, rx, rc, sx, sc, delta_w=1e-3)
    inert = prob.kkt_factor(x, given, hes, sig, delta_w=1e-3)
    assert abs(sd - inert.schur_d) <= 1e-12 * abs(sd)
    h = lambda t: t.cpu().numpy()  # noqa: E731
    dz, dd = prob.from_soa(h(sx))
    dl, _ = prob.from_soa(h(sc))
    args = prob.values_to_scen(h(hes), len(hr)), prob.from_soa(h(sig))[0], prob.from_soa(h(rx))[0], prob.from_soa(h(rc))[0]
    for s in list(seen)[:8]:
        z, c = _residual(prob, J, *args, dz, dl, dd, 1e-3, jr, jc, hr, hc, s)
        assert z <= 1e-12 and c <= 1e-12, s
    # the evaluation's own values again: nothing of the other factors is left behind
    again = torch.zeros_like(rx), torch.zeros_like(rc)
    B.kkt_newton_noalloc(P, S, prob.ld, x, jac, hes, sig, rx, rc, *again, delta_w=1e-3)
    assert torch.equal(own[0], again[0]) and torch.equal(own[1], again[1])
