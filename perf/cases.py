"""Workloads of the absorber library, through its public binding.

One case is one call that a user's program makes: the fused evaluation, a Newton direction
(kkt_factor + kkt_solve), an interior-point solve, or a pass of the warm-start network.
Sizes are the scenario counts of the repository's workloads (10 to 20,000 scenarios, a batch
of problems with 50 to 2000 scenarios each) and the row counts the network meets.

Inputs of the evaluation and of the Newton directions are iterates of the middle of a solve:
the column profile below (the nominal feed's converged stage states), every entry perturbed
per scenario, with barrier terms of mu = 1e-2.  Derivatives, right-hand sides and the values
of exact() come from the model equations written in torch here, differentiated by autograd in
64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import absorber_inputs as ai
from paper_2607_15420_gb300 import binding as B

P = ai.PARAMS
N, NV = 10, 22
NLOC = 40                     # local quantities of a stage's rows: own 22, above 11, below 6, d
ABOVE = tuple(range(9)) + (13, 15)           # stage n+1's unknowns a stage reads: x, L, T
BELOW = (9, 10, 11, 12, 14, 15)              # stage n-1's: y, V, T
MU = 1e-2
DIAMETER = 1.8

# stage states of the nominal feed at its optimum, bottom to top: 9 scaled liquid fractions,
# 4 vapour fractions, L, V, T / 100, 5 extents
PROFILE = (
    (0.01728685, 4.923845, 12.90198, 4.591562, 3.222989, 0.4315847, 0.4970273, 29.34604, 0.8842566, 0.08613628,
     0.1710084, 0.6970001, 0.04585527, 0.4476331, 0.1090387, 3.335571, -0.002602753, 1.102911e-06, -1.893534e-07,
     -0.002171708, 0.002601839),
    (0.02724438, 4.232336, 10.85518, 4.002329, 2.207155, 0.8329347, 0.4604156, 15.60152, 0.8881393, 0.0530021,
     0.2485654, 0.6553194, 0.04311312, 0.4592736, 0.115974, 3.41787, -0.003241219, 2.677213e-07, -3.360039e-07,
     -0.002884623, 0.003241287),
    (0.03970276, 3.450161, 7.631217, 3.3011, 1.400131, 1.530618, 0.444732, 6.661995, 0.8913318, 0.02445145,
     0.3028502, 0.6311738, 0.04152459, 0.4694502, 0.1204106, 3.462924, -0.003200164, -1.56181e-07, -5.064877e-07,
     -0.002967714, 0.003200827),
    (0.05199537, 2.724158, 5.012715, 2.626206, 0.8887729, 2.567739, 0.4408862, 2.729936, 0.8935628, 0.010318,
     0.3264699, 0.6222731, 0.04093902, 0.4770876, 0.1221329, 3.480137, -0.001682974, -1.766875e-07, -3.830659e-07,
     -0.001591323, 0.001683534),
    (0.05844127, 2.354589, 3.90198, 2.276406, 0.6901974, 3.346773, 0.4414383, 1.645016, 0.8945094, 0.006244752,
     0.3301983, 0.6225966, 0.0409603, 0.4804934, 0.1220694, 3.482594, -0.0004974484, -1.606306e-07, -1.293398e-07,
     -0.0004697645, 0.0004977384),
    (0.06039963, 2.249028, 3.518119, 2.176672, 0.6310736, 3.612689, 0.4443797, 1.361733, 0.8946629, 0.005127132,
     0.3234146, 0.6300102, 0.04144804, 0.4809277, 0.120633, 3.477604, -0.0001433541, -3.275418e-07, -2.02474e-08,
     -0.0001258502, 0.0001437019),
    (0.0611237, 2.225202, 3.183175, 2.1563, 0.5948724, 3.66464, 0.4524064, 1.177476, 0.8944163, 0.004319811,
     0.3027887, 0.6501204, 0.04277108, 0.479635, 0.1169014, 3.462062, -0.0001125711, -8.141476e-07, 2.027539e-08,
     -8.258588e-05, 0.0001133649),
    (0.06199827, 2.218467, 2.574294, 2.15534, 0.5330241, 3.649901, 0.4729484, 0.8834709, 0.8936788, 0.003036055,
     0.2563854, 0.6948639, 0.04571473, 0.4760168, 0.1093739, 3.423548, -0.0001709689, -1.82785e-06, 6.128193e-08,
     -0.0001205392, 0.0001727355),
    (0.06359322, 2.216801, 1.655679, 2.163444, 0.4261156, 3.57642, 0.5193719, 0.489401, 0.8921222, 0.001463258,
     0.179667, 0.7683223, 0.05054752, 0.468662, 0.09891683, 3.344378, -0.000184199, -3.09918e-06, 1.102202e-07,
     -0.0001306097, 0.000187188),
    (0.06570474, 2.226283, 0.8512458, 2.183422, 0.3054737, 3.416097, 0.5986179, 0.2024411, 0.8898293, 0.0004888475,
     0.1037336, 0.8404826, 0.05529491, 0.4583921, 0.09042424, 3.229875, -9.738378e-05, -3.214428e-06, 1.124494e-07,
     -6.599471e-05, 0.0001004858),
)

PRECISION = {"fp64": B.PREC_FP64, "fp32": B.PREC_FP32, "ldl": B.PREC_FP64_LDL}


def listed():
    return [
        # one evaluation of a study of a few scenarios (a ragged second warp): launch latency
        {"name": "eval-33", "kind": "eval", "S": 33, "out": "hess"},
        # residuals and Jacobian alone, as a user's own solver or a sensitivity study asks for
        {"name": "eval-jac-500", "kind": "eval", "S": 500, "out": "jac"},
        # the evaluation of every iteration at the headline size
        {"name": "eval-5000", "kind": "eval", "S": 5000, "out": "hess"},
        # Newton directions, the KKT step of one iteration: the ten-scenario problem ...
        {"name": "newton-fp64-10", "kind": "newton", "S": 10, "prec": "fp64", "delta_w": 0.0, "delta_c": 0.0},
        # ... the 500-scenario one, with a primal regularisation ...
        {"name": "newton-fp64-500", "kind": "newton", "S": 500, "prec": "fp64", "delta_w": 1e-4, "delta_c": 0.0},
        # ... mixed precision at the headline size (FP32 factors, refinement in FP64) ...
        {"name": "newton-fp32-5000", "kind": "newton", "S": 5000, "prec": "fp32", "delta_w": 0.0, "delta_c": 0.0},
        # ... the largest workload in FP64 ...
        {"name": "newton-fp64-20000", "kind": "newton", "S": 20000, "prec": "fp64", "delta_w": 0.0, "delta_c": 0.0},
        # ... and the dual-regularised system (block LDL^T) of a nearly singular iterate
        {"name": "newton-ldl-500", "kind": "newton", "S": 500, "prec": "ldl", "delta_w": 0.0, "delta_c": 1e-6},
        # the warm-start network's prediction for every scenario of the headline problem
        {"name": "network-forward-5000", "kind": "forward", "n": 5000},
        # one training minibatch of it (the default batch): loss and gradient
        {"name": "network-gradient-512", "kind": "gradient", "n": 512},
        # a whole interior-point solve from the default start: the headline problem
        {"name": "solve-fp32-5000", "kind": "solve", "S": 5000, "prec": "fp32"},
        # a batch of 64 independent problems of 50 to 2000 scenarios
        {"name": "batch-fp32-64", "kind": "batch", "P": 64, "lo": 50, "hi": 2000, "prec": "fp32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("eval", "eval", "newton", "newton", "newton", "forward", "gradient", "solve", "batch"))
    if kind == "eval":
        return {"kind": kind, "S": _log(rng, 1, 20000), "out": rng.choice(("hess", "hess", "jac", "c"))}
    if kind == "newton":
        prec = rng.choice(("fp64", "fp32", "fp64", "fp32", "ldl"))
        return {"kind": kind, "S": _log(rng, 1, 500 if prec == "ldl" else 20000), "prec": prec,
                "delta_w": rng.choice((0.0, 1e-4)), "delta_c": rng.choice((1e-8, 1e-6)) if prec == "ldl" else 0.0}
    if kind in ("forward", "gradient"):
        return {"kind": kind, "n": _log(rng, 1, 20000) if kind == "forward" else _log(rng, 32, 4096)}
    prec = rng.choice(("fp64", "fp32"))
    if kind == "solve":
        return {"kind": kind, "S": _log(rng, 10, 5000), "prec": prec}
    return {"kind": kind, "P": _log(rng, 4, 64), "lo": 50, "hi": _log(rng, 100, 1000), "prec": prec}


# ---- the model in torch ------------------------------------------------------------------


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (seed % 65_521) + 17)
    return g


def _feeds(S, seed):
    return ai.make_feeds(S, seed % (1 << 31))


def _stage_rows(q, pres):
    """The 22 rows of a stage; q: 40 local quantities, each [10, S]; pres [10, S]."""
    sx, sy, sT = P["sx"], P["sy"], P["sT"]
    nu = ((0, (1, 0, 0, 1, 0)), (1, (-1, 0, 0, 0, 0)), (2, (1, 1, 1, 0, 1)), (3, (0, 0, 0, -1, 0)),
          (4, (0, -1, 0, 1, 1)), (5, (0, 0, 1, 0, 0)), (6, (0, 1, 0, 0, 0)), (7, (0, 0, 0, 0, -1)),
          (8, (0, 0, -1, -1, -1)))
    nu = dict(nu)
    x, y = [sx[i] * q[i] for i in range(9)], [sy[j] * q[9 + j] for j in range(4)]
    L, V, T, eps = q[13], q[14], sT * q[15], q[16:21]
    xa, La, Ta = [sx[i] * q[22 + i] for i in range(9)], q[31], sT * q[32]
    yb, Vb, Tb = [sy[j] * q[33 + j] for j in range(4)], q[37], sT * q[38]

    def h(kind, i, t):
        dt = t - P["T_ref"]
        return P[kind + "_ref"][i] + P[kind + "_dh"][i] + dt * (P[kind + "_cpa"][i] + 0.5 * P[kind + "_cpb"][i] * dt)

    rows = []
    for c in range(11):
        r = torch.zeros_like(L)
        if c < 9:
            r = r + L * x[c] - La * xa[c]
            for k in range(5):
                if nu[c][k]:
                    r = r - nu[c][k] * eps[k]
        if c >= 7:
            r = r + V * y[c - 7] - Vb * yb[c - 7]
        rows.append(r)
    rows.append(pres * y[1] - x[8] * torch.exp(P["psat_a"] - P["psat_b"] / (T + P["psat_c"])))
    am, ac, aw = x[0] + x[1] + x[3], x[7] + x[3] + x[4] + x[6], x[8] + x[4] + x[6] + x[5]
    tot = am + ac + aw
    lnh = P["henry_a"] + P["henry_b"] / T + P["henry_m"] * (am / tot) + P["henry_w"] * (aw / tot)
    rows.append(pres * y[0] - P["rho_L"] * x[7] * torch.exp(lnh))
    for k in range(5):
        r = -(P["KE_A"][k] + P["KE_B"][k] / T + P["KE_C"][k] * torch.log(T) + P["KE_D"][k] * T)
        for c in range(9):
            if nu[c][k]:
                r = r + nu[c][k] * (torch.log(q[c]) + math.log(sx[c]))
        rows.append(r)
    rows.append(sum(x) - 1.0)
    rows.append(sum(y) - 1.0)
    rows.append(L * sum(x[i] * h("hL", i, T) for i in range(9)) + V * sum(y[j] * h("hV", j, T) for j in range(4))
                - La * sum(xa[i] * h("hL", i, Ta) for i in range(9)) - Vb * sum(yb[j] * h("hV", j, Tb) for j in range(4)))
    rows.append(V * P["R"] * T / pres - P["u_max"] * math.pi * q[39] * q[39] / 4.0 + q[21])
    return rows


def _local(Z, d, F):
    """The 40 local quantities [40, 10, S] of every stage; Z [10, 22, S], F [18, S]."""
    S = Z.shape[2]
    q = torch.empty((NLOC, N, S), dtype=torch.float64, device="cuda")
    q[:NV] = Z.permute(1, 0, 2)
    for a, j in enumerate(ABOVE):
        q[22 + a, :N - 1] = Z[1:, j]
    for i in range(9):
        q[22 + i, N - 1] = F[7 + i] / P["sx"][i]
    q[31, N - 1], q[32, N - 1] = F[6], F[16] / P["sT"]
    for b, j in enumerate(BELOW):
        q[33 + b, 1:] = Z[:N - 1, j]
    for j in range(4):
        q[33 + j, 0] = F[1 + j] / P["sy"][j]
    q[37, 0], q[38, 0] = F[0], F[5] / P["sT"]
    q[39] = d
    return q


def _columns(rows, cols):
    """Stage, row and local quantity of every pattern entry."""
    n, r, loc = rows // NV, rows % NV, []
    for i, (row, col) in enumerate(zip(rows, cols)):
        k, j = col // NV, col % NV
        loc.append(39 if col == N * NV else j if k == n[i] else 22 + ABOVE.index(j) if k > n[i] else 33 + BELOW.index(j))
    return tuple(torch.as_tensor(np.asarray(v, dtype=np.int64), device="cuda") for v in (n, r, loc))


def _derivatives(Z, d, F, lam, want):
    """Residuals [220, S], Jacobian and Hessian values in pattern order [nnz, S] (or None)."""
    S = Z.shape[2]
    pres = F[17][None, :].expand(N, S)
    q = _local(Z, d, F)
    jr, jc, hr, hc = B.scenario_pattern()
    qs = [v.clone().requires_grad_(want != "c") for v in q]
    rows = _stage_rows(qs, pres)
    c = torch.stack([r.detach() for r in rows]).permute(1, 0, 2).reshape(N * NV, S)
    J = H = None
    if want in ("jac", "hess"):
        Jl = torch.zeros((NV, NLOC, N, S), dtype=torch.float64, device="cuda")
        for r, row in enumerate(rows):
            for i, v in enumerate(torch.autograd.grad(row.sum(), qs, retain_graph=True, allow_unused=True)):
                if v is not None:
                    Jl[r, i] = v
        n, r, loc = _columns(jr, jc)
        J = Jl[r, loc, n]
        del Jl
    if want == "hess":
        lg = sum((l * row).sum() for l, row in zip(lam.view(N, NV, S).permute(1, 0, 2), rows))
        first = torch.autograd.grad(lg, qs, create_graph=True, allow_unused=True)
        W = torch.zeros((N, NV, NV, S), dtype=torch.float64, device="cuda")
        Wd = torch.zeros(S, dtype=torch.float64, device="cuda")

        def second(i, others):
            if first[i] is None or not first[i].requires_grad:
                return [None] * len(others)
            return torch.autograd.grad(first[i].sum(), [qs[k] for k in others], retain_graph=True, allow_unused=True)

        for j in range(NV):
            for k, v in enumerate(second(j, range(NV))):
                if v is not None:
                    W[:, j, k] += v
        for off, var, to, frm in ((22, ABOVE, slice(1, N), slice(0, N - 1)), (33, BELOW, slice(0, N - 1), slice(1, N))):
            for a, j in enumerate(var):
                for b, v in enumerate(second(off + a, [off + k for k in range(len(var))])):
                    if v is not None:
                        W[to, j, var[b]] += v[frm]
        v = second(39, [39])[0]
        if v is not None:
            Wd += v.sum(0)
        last = len(hr) - 1
        n = torch.as_tensor(hr[:last] // NV, device="cuda", dtype=torch.int64)
        H = torch.empty((len(hr), S), dtype=torch.float64, device="cuda")
        H[:last] = W[n, torch.as_tensor(hr[:last] % NV, device="cuda", dtype=torch.int64),
                     torch.as_tensor(hc[:last] % NV, device="cuda", dtype=torch.int64)]
        H[last] = Wd
    return c, J, H


def _iterate(S, seed):
    """A mid-solve iterate: feeds (host and device), stage states Z [10, 22, S], d, multipliers."""
    g = _generator(seed)
    Fh = _feeds(S, seed)
    F = torch.from_numpy(Fh).cuda()
    rnd = lambda *shape: torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    base = torch.tensor(PROFILE, dtype=torch.float64, device="cuda")
    Z = torch.empty((N, NV, S), dtype=torch.float64, device="cuda")
    Z[:, :15] = base[:, :15, None] * torch.exp(0.05 * rnd(N, 15, S))
    Z[:, 15] = base[:, 15, None] + 0.01 * rnd(N, S)
    Z[:, 16:21] = base[:, 16:21, None] * (1.0 + 0.1 * rnd(N, 5, S))
    Z[:, 21] = P["u_max"] * math.pi * DIAMETER ** 2 / 4.0 - Z[:, 14] * P["R"] * P["sT"] * Z[:, 15] / F[17]
    lam = 0.1 * rnd(N, NV, S)
    lam[:, 21] = MU / Z[:, 21] * torch.exp(0.3 * rnd(N, S))
    return Fh, F, Z, lam.reshape(N * NV, S), rnd


def _pad(v, ld, tail=None):
    """[k, S] -> flat structure of arrays with leading dimension ld (and the design entry)."""
    out = torch.zeros((v.shape[0], ld), dtype=torch.float64, device="cuda")
    out[:, :v.shape[1]] = v
    out = out.view(-1)
    return out if tail is None else torch.cat([out, torch.tensor([float(tail)], dtype=torch.float64, device="cuda")])


def _newton_system(S, seed):
    """A Newton system: iterate, derivatives, barrier diagonal and right-hand sides."""
    Fh, F, Z, lam, rnd = _iterate(S, seed)
    c, J, H = _derivatives(Z, DIAMETER, F, lam, "hess")
    jr, jc, _, _ = B.scenario_pattern()
    jr, jc = (torch.as_tensor(v, device="cuda", dtype=torch.int64) for v in (jr, jc))
    x = Z.reshape(N * NV, S)
    lo = torch.zeros((N, NV), dtype=torch.float64, device="cuda")
    lo[:, 15] = P["T_lo"] / P["sT"]
    has = torch.ones((N, NV), dtype=torch.bool, device="cuda")
    has[:, 16:21] = False
    sl = torch.where(has.view(-1, 1), x - lo.view(-1, 1), torch.ones_like(x))
    z = torch.where(has.view(-1, 1), MU / sl * torch.exp(0.3 * rnd(N * NV, S)), torch.zeros_like(x))
    sig, gb = z / sl, torch.where(has.view(-1, 1), -MU / sl, torch.zeros_like(x))
    hot = torch.zeros((N, NV), dtype=torch.bool, device="cuda")
    hot[:, 15] = True
    su = torch.where(hot.view(-1, 1), P["T_hi"] / P["sT"] - x, torch.ones_like(x))
    sig = sig + torch.where(hot.view(-1, 1), MU / su ** 2, torch.zeros_like(x))
    gb = gb + torch.where(hot.view(-1, 1), MU / su, torch.zeros_like(x))
    JT = torch.zeros((N * NV + 1, S), dtype=torch.float64, device="cuda").index_add_(0, jc, J * lam[jr])
    dl, du = DIAMETER - P["d_lo"], P["d_hi"] - DIAMETER
    rd = -(S + float(JT[-1].sum()) - MU / dl + MU / du)   # the objective is scaled by S
    return {"feeds": Fh, "x": x, "jac": J, "hess": H, "sig": sig, "sigd": MU / dl ** 2 + MU / du ** 2,
            "rz": -(JT[:-1] + gb), "rd": rd, "rc": -c}


# ---- the network's inputs ------------------------------------------------------------------

WIDTHS = ((3, 256), (256, 256), (256, 256), (256, 440))


def _network_inputs(n, seed):
    g = _generator(seed)
    rnd = lambda *shape: torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)  # noqa: E731
    theta = torch.cat([v for i, o in WIDTHS for v in (rnd(o * i) * math.sqrt(2.0 / (i + o)), 0.1 * rnd(o))])
    shift, scale = np.array([0.10, 0.12, 1.5]), np.array([0.0058, 0.0069, 0.08])
    f = torch.from_numpy(_feeds(n, seed)[[0, 1]]).cuda().to(torch.float32)
    X = torch.stack([f[0], f[1], 1.5 + 0.08 * rnd(n)], dim=1).contiguous()
    oshift, oscale = rnd(440), torch.exp(0.5 * rnd(440))
    Y = (oshift + oscale * rnd(n, 440)).contiguous()
    return theta, shift, scale, oshift, oscale, X, Y


# ---- prepare, run ----------------------------------------------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    if kind == "eval":
        S = case["S"]
        Fh, F, Z, lam, _ = _iterate(S, seed)
        p = B.Problem(P, Fh)
        new = lambda n: torch.zeros(n * p.ld, dtype=torch.float64, device="cuda")  # noqa: E731
        return {"kind": kind, "p": p, "S": S, "x": _pad(Z.reshape(-1, S), p.ld, DIAMETER), "lam": _pad(lam, p.ld),
                "c": new(N * NV), "jac": new(p.sizes.nnzJ_scen) if case["out"] != "c" else None,
                "hess": new(p.sizes.nnzH_scen) if case["out"] == "hess" else None}
    if kind == "newton":
        S = case["S"]
        s = _newton_system(S, seed)
        p = B.Problem(P, s["feeds"])
        st = {"kind": kind, "p": p, "S": S, "x": _pad(s["x"], p.ld, DIAMETER), "jac": _pad(s["jac"], p.ld),
              "hess": _pad(s["hess"], p.ld), "sig": _pad(s["sig"], p.ld, s["sigd"]),
              "rx": _pad(s["rz"], p.ld, s["rd"]), "rc": _pad(s["rc"], p.ld), "prec": PRECISION[case["prec"]],
              "delta_w": case["delta_w"], "delta_c": case["delta_c"],
              # the refinement a direction to full accuracy needs: the binding's two rounds for
              # FP64 factors, more for FP32 ones
              "refine": 8 if case["prec"] == "fp32" else 2}
        st["sx"], st["sc"] = torch.zeros_like(st["rx"]), torch.zeros_like(st["rc"])
        return st
    if kind in ("forward", "gradient"):
        theta, shift, scale, oshift, oscale, X, Y = _network_inputs(case["n"], seed)
        net = B.MLP(1)
        net.set_params(theta.cpu().numpy())
        net.set_normalization(shift, scale, oshift.cpu().numpy(), oscale.cpu().numpy())
        out = torch.zeros(B.MLP_PARAMS, device="cuda") if kind == "gradient" else torch.zeros_like(Y)
        return {"kind": kind, "net": net, "X": X, "Y": Y, "out": out}
    o = B.default_options(**({"precision": B.PREC_FP32, "max_refine": 8} if case["prec"] == "fp32" else {}))
    if kind == "solve":
        p = B.Problem(P, _feeds(case["S"], seed))
    else:
        sizes = ai.batched_sizes(case["P"], 3, case["lo"], case["hi"])
        p = B.Batch(P, ai.batched_feeds(sizes, seed % (1 << 31)))
    return {"kind": kind, "p": p, "S": p.S, "o": o, "x": torch.zeros(p.n_primal, dtype=torch.float64, device="cuda"),
            "y": torch.zeros(p.n_row, dtype=torch.float64, device="cuda")}


def _live(v, st, rows):
    """The scenarios of a flat vector, without the padding (whose contents are unspecified)."""
    ld = st["p"].ld
    return v[:rows * ld].view(rows, ld)[:, :st["S"]]


def run(st):
    kind = st["kind"]
    if kind == "eval":
        st["p"].eval_grad_jac_hess(st["x"], st["lam"], 1.0, c=st["c"], jac=st["jac"], hess=st["hess"])
        z = st["p"].sizes
        return {"c": _live(st["c"], st, N * NV), "jac": None if st["jac"] is None else _live(st["jac"], st, z.nnzJ_scen),
                "hess": None if st["hess"] is None else _live(st["hess"], st, z.nnzH_scen)}
    if kind == "newton":
        i = st["p"].kkt_factor(st["x"], st["jac"], st["hess"], st["sig"], delta_w=st["delta_w"],
                               delta_c=st["delta_c"], precision=st["prec"])
        st["p"].kkt_solve(st["rx"], st["rc"], st["sx"], st["sc"], max_refine=st["refine"])
        return {"dz": _live(st["sx"], st, N * NV), "dd": st["sx"][-1:], "dl": _live(st["sc"], st, N * NV),
                "inertia": [int(i.n_pos), int(i.n_neg), int(i.n_zero), int(i.n_singular)]}
    if kind == "forward":
        st["net"].forward(st["X"], st["out"])
        return st["out"]
    if kind == "gradient":
        loss = st["net"].loss_grad(st["X"], st["Y"], st["out"])
        return {"loss": loss, "grad": st["out"]}
    r = st["p"].ipm_solve(st["o"], x_out=st["x"], y_out=st["y"])
    r = r if isinstance(r, list) else [r]
    return {"x": _live(st["x"], st, N * NV), "y": _live(st["y"], st, N * NV),
            "d": st["x"][N * NV * st["p"].ld:][:len(r)], "status": np.array([v.status for v in r])}


# ---- what a pass cannot do without ------------------------------------------------------------


def work(case):
    kind = case["kind"]
    jr, _, hr, _ = B.scenario_pattern()
    nj, nh, v = len(jr), len(hr), N * NV
    if kind == "eval":
        out = {"c": v, "jac": v + nj, "hess": v + nj + nh}[case["out"]]
        read = v + 18 + (v if case["out"] == "hess" else 0)
        flops = {"c": 9_900, "jac": 13_000, "hess": 19_000}[case["out"]]   # the stage equations of a scenario
        return {"bytes": 8 * case["S"] * (read + out), "flops": flops * case["S"]}
    # a direction reads the derivatives, the barrier diagonal and the right-hand sides once and
    # writes the direction; its arithmetic: the sparse residual of the system, twice
    newton = {"bytes": 8 * (nj + nh + v + 4 * v), "flops": 2 * 2 * (2 * nj + 2 * nh)}
    if kind == "newton":
        return {k: case["S"] * n for k, n in newton.items()}
    if kind == "forward":
        return {"bytes": 4 * case["n"] * 443 + 2 * B.MLP_PARAMS, "flops": 2 * case["n"] * (B.MLP_PARAMS - 1208)}
    if kind == "gradient":
        return {"bytes": 4 * case["n"] * 443 + 6 * B.MLP_PARAMS, "flops": 6 * case["n"] * (B.MLP_PARAMS - 1208)}
    # a solve: about 30 iterations of an evaluation and a direction
    S = case["S"] if kind == "solve" else case["P"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
    step = {"bytes": newton["bytes"] + 8 * (2 * v + 18 + v + nj + nh), "flops": newton["flops"] + 19_000}
    return {k: 30 * S * n for k, n in step.items()}


# ---- the outputs in 64 bits ---------------------------------------------------------------------


def _exact_newton(case, seed):
    S = case["S"]
    s = _newton_system(S, seed)
    jr, jc, hr, hc = (torch.as_tensor(a, device="cuda", dtype=torch.int64) for a in B.scenario_pattern())
    nz, dw, dc = N * NV, case["delta_w"], case["delta_c"]
    dz, dl = torch.empty((nz, S), dtype=torch.float64, device="cuda"), torch.empty((nz, S), dtype=torch.float64, device="cuda")
    uz, ul = torch.empty_like(dz), torch.empty_like(dl)
    Sd = float(s["hess"][-1].sum()) + s["sigd"] + dw
    rd = s["rd"]
    for a in range(0, S, 500):     # dense 440 x 440 systems, a block of scenarios at a time
        e = min(S, a + 500)
        J = torch.zeros((e - a, nz, nz + 1), dtype=torch.float64, device="cuda")
        J[:, jr, jc] = s["jac"][:, a:e].T
        H = torch.zeros((e - a, nz, nz), dtype=torch.float64, device="cuda")
        H[:, hr[:-1], hc[:-1]] = s["hess"][:-1, a:e].T
        H[:, hc[:-1], hr[:-1]] = s["hess"][:-1, a:e].T
        H.diagonal(dim1=1, dim2=2).add_(s["sig"][:, a:e].T + dw)
        b, J = J[:, :, nz], J[:, :, :nz]
        K = torch.zeros((e - a, 2 * nz, 2 * nz), dtype=torch.float64, device="cuda")
        K[:, :nz, :nz], K[:, :nz, nz:], K[:, nz:, :nz] = H, J.transpose(1, 2), J
        K[:, nz:, nz:].diagonal(dim1=1, dim2=2).fill_(-dc)
        rhs = torch.zeros((e - a, 2 * nz, 2), dtype=torch.float64, device="cuda")
        rhs[:, :nz, 0], rhs[:, nz:, 0], rhs[:, nz:, 1] = s["rz"][:, a:e].T, s["rc"][:, a:e].T, b
        LU, piv = torch.linalg.lu_factor(K)
        v = torch.linalg.lu_solve(LU, piv, rhs)
        for _ in range(2):
            v = v + torch.linalg.lu_solve(LU, piv, rhs - K @ v)
        Sd -= float((b * v[:, nz:, 1]).sum())
        rd -= float((b * v[:, nz:, 0]).sum())
        dz[:, a:e], dl[:, a:e], uz[:, a:e], ul[:, a:e] = v[:, :nz, 0].T, v[:, nz:, 0].T, v[:, :nz, 1].T, v[:, nz:, 1].T
    dd = rd / Sd
    return {"dz": dz - uz * dd, "dd": torch.tensor([dd], dtype=torch.float64, device="cuda"), "dl": dl - ul * dd,
            "inertia": [None] * 4}


def _exact_network(case, seed):
    theta, shift, scale, oshift, oscale, X, Y = _network_inputs(case["n"], seed)
    W, b, at = [], [], 0
    for i, o in WIDTHS:
        # the network's weights are the bfloat16 roundings of its parameters
        W.append(theta[at:at + i * o].to(torch.bfloat16).double().view(o, i).requires_grad_(True))
        b.append(theta[at + i * o:at + i * o + o].double().requires_grad_(True))
        at += i * o + o
    f = lambda v: torch.as_tensor(v, device="cuda").to(torch.float32).double()  # noqa: E731
    a = (X.double() - f(shift)) / f(scale)
    for l in range(4):
        a = a @ W[l].T + b[l]
        a = a * 0.5 * (1.0 + torch.erf(a / math.sqrt(2.0))) if l < 3 else a
    if case["kind"] == "forward":
        return (a * f(oscale) + f(oshift)).detach()
    loss = ((a - (Y.double() - f(oshift)) / f(oscale)) ** 2).sum() / (2.0 * a.numel())
    loss.backward()
    return {"loss": float(loss.detach()), "grad": torch.cat([v.grad.reshape(-1) for p in zip(W, b) for v in p])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "eval":
        _, F, Z, lam, _ = _iterate(case["S"], seed)
        c, J, H = _derivatives(Z, DIAMETER, F, lam, case["out"])
        return {"c": c, "jac": J, "hess": H}
    if kind == "newton":
        # a dense factorization of every scenario's 440 x 440 system: minutes at 20,000
        return _exact_newton(case, seed) if case["S"] <= 5000 else None
    if kind in ("forward", "gradient"):
        return _exact_network(case, seed)
    return None   # an interior-point solve: its own tolerance decides where it stops
