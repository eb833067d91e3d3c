// model.cuh -- the absorber stage equations of the case study with analytic first and
// second derivatives, for one (scenario, stage).  __host__ __device__: the device
// kernels evaluate values with it, and the host runs the same routine once per stage
// type with a recording emitter to derive the sparsity pattern, so the pattern and
// the values written by the kernel come from one piece of code.
//
// Equations (paper, Sections "Equilibrium process model" and "Case study"):
//   (1)  material balance  L x_i + V y_i - L+ x_i+ - V- y_i- - sum_r nu_ir eps_r = 0
//   (9a) Raoult (water)    P y_H2O - x_H2O Psat(T) = 0
//   (9b) Henry (CO2)       P y_CO2 - rho_L x_CO2 H(T, x_MEA^app, x_H2O^app) = 0
//   (3a) reaction equil.   sum_i nu_ir ln x_i - ln K_r(T) = 0,  activities = x
//   (4)  summation         sum x - 1 = 0,  sum y - 1 = 0
//   (6)  energy balance    L h^L + V h^V - L+ h^L+ - V- h^V- = 0 (ideal mixtures, Q = 0)
//   (10b) hydraulic        V R T / P - u_max pi d^2 / 4 + s = 0,  s >= 0
// with Kent-Eisenberg ln K_r = A + B/T + C ln T + D T, Antoine ln Psat = a - b/(T+c),
// ln H = ha + hb/T + hm x_MEA^app + hw x_H2O^app, apparent fractions normalised over
// (MEA, CO2, H2O)_app, and h_i(T) = ref + cpa (T-Tref) + cpb/2 (T-Tref)^2 + dh.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifndef __CUDACC__
#define __host__
#define __device__
#endif

namespace absorber {

constexpr int N_STAGES = 10;
constexpr int NV = 22;          // unknowns per stage
constexpr int NR = 22;          // rows per stage
constexpr int NSC = N_STAGES * NV;  // unknowns (= rows) per scenario
constexpr int NLOC = 40;        // local variables of one stage's rows
constexpr int NFEED = 18;

// local-variable numbering of one stage's rows
constexpr int LX = 0, LY = 9, LL = 13, LV = 14, LT = 15, LE = 16, LS = 21;
constexpr int AX = 22, AL = 31, AT = 32;     // stream from above (stage n+1)
constexpr int BY = 33, BV = 37, BT = 38;     // stream from below (stage n-1)
constexpr int LD_ = 39;                      // the diameter
// rows
constexpr int R_VH = 11, R_VC = 12, R_RX = 13, R_SX = 18, R_SY = 19, R_E = 20, R_H = 21;

// feed record offsets
constexpr int F_V0 = 0, F_Y0 = 1, F_T0 = 5, F_LIN = 6, F_XIN = 7, F_TIN = 16, F_P = 17;

// stoichiometry nu[species][reaction] of R1..R5; species MEA, MEAH+, H+, MEACOO-,
// HCO3-, OH-, CO3--, CO2, H2O, N2, O2
__host__ __device__ constexpr int nu(int c, int r) {
    // R1: MEAH+ -> MEA + H+ ; R2: HCO3- -> H+ + CO3-- ; R3: H2O -> H+ + OH- ;
    // R4: MEACOO- + H2O -> MEA + HCO3- ; R5: H2O + CO2 -> H+ + HCO3-
    constexpr int t[11][5] = {
        {1, 0, 0, 1, 0},     // MEA
        {-1, 0, 0, 0, 0},    // MEAH+
        {1, 1, 1, 0, 1},     // H+
        {0, 0, 0, -1, 0},    // MEACOO-
        {0, -1, 0, 1, 1},    // HCO3-
        {0, 0, 1, 0, 0},     // OH-
        {0, 1, 0, 0, 0},     // CO3--
        {0, 0, 0, 0, -1},    // CO2
        {0, 0, -1, -1, -1},  // H2O
        {0, 0, 0, 0, 0},     // N2
        {0, 0, 0, 0, 0},     // O2
    };
    return t[c][r];
}

// membership of the liquid species in the apparent MEA / CO2 / H2O totals of (9b)
__host__ __device__ constexpr int app_m(int k) { return (k == 0 || k == 1 || k == 3) ? 1 : 0; }
__host__ __device__ constexpr int app_c(int k) { return (k == 7 || k == 3 || k == 4 || k == 6) ? 1 : 0; }
__host__ __device__ constexpr int app_w(int k) { return (k == 8 || k == 4 || k == 6 || k == 5) ? 1 : 0; }
__host__ __device__ constexpr int app_t(int k) { return app_m(k) + app_c(k) + app_w(k); }
__host__ __device__ constexpr bool in_henry(int k) { return app_t(k) > 0; }

struct Params {
    double R, u_max, d_lo, d_hi, T_lo, T_hi, T_ref;
    double sx[9], sy[4], sT;
    double KE_A[5], KE_B[5], KE_C[5], KE_D[5];
    double psat_a, psat_b, psat_c;
    double henry_a, henry_b, henry_m, henry_w, rho_L;
    double hL_ref[9], hL_cpa[9], hL_cpb[9], hL_dh[9];
    double hV_ref[4], hV_cpa[4], hV_cpb[4], hV_dh[4];
    int nsec;        // column sections, each with its own diameter (1 or 2)
    double dp_stage; // specified pressure drop per stage (relation (7)); 0: P^abs everywhere
    // derived at creation
    double lnsx[9];
    double lnsxr[5];   // sum_c nu_ck ln sx_c: the scales' share of each reaction's quotient
    double hL0[9];   // hL_ref + hL_dh
    double hV0[4];
    double Tlo_s, Thi_s;   // T_lo / sT, T_hi / sT: the scaled temperature bounds
    double sxx[45];        // sx_k sx_l, l <= k, at k (k + 1) / 2 + l
};

// The species of the apparent totals fall into five classes of equal membership (MEA, MEAH+ |
// MEACOO- | HCO3-, CO3-- | OH-, H2O | CO2): Henry's derivatives are formed once per class.
// c_t: totals the class counts in; c_a: 1 MEA, 2 H2O, 0 neither.
__host__ __device__ constexpr int henry_cls(int k) {
    constexpr int t[9] = {0, 0, -1, 1, 2, 3, 2, 4, 3};
    return t[k];
}
__host__ __device__ constexpr int cls_t(int c) { return c == 1 || c == 2 ? 2 : 1; }
__host__ __device__ constexpr int cls_a(int c) { return c < 2 ? 1 : (c < 4 ? 2 : 0); }

constexpr int KSEC = 2;   // most column sections (design-vector entries)

// the section of stage n among K: consecutive stages, floor(n K / N)
__host__ __device__ constexpr int stage_sec(int n, int K) { return (n * K) / N_STAGES; }

// objective weight of section k's diameter: its share of the stages
__host__ __device__ inline double sec_weight(int k, int K) {
    int c = 0;
    for (int n = 0; n < N_STAGES; ++n) c += stage_sec(n, K) == k ? 1 : 0;
    return (double)c / N_STAGES;
}

// pressure of stage n by relation (7) with a specified drop, Pt the top stage's
__host__ __device__ inline double stage_pres(const Params& P, double Pt, int n) {
    return Pt + (double)(N_STAGES - 1 - n) * P.dp_stage;
}

struct StageIn {
    double q[NV];     // own scaled unknowns
    double qa[11];    // from above, in physical units: x[9], L, T  (the lean feed on the top stage)
    double qb[6];     // from below: y[4], V, T  (the flue gas on stage 0)
    double d, P;
    bool has_above, has_below;   // neighbour stage exists (its values are unknowns)
};

struct StageLam {
    double own[NR];
    double below[10];   // stage n-1: material multipliers of the 9 liquid species, energy
    double above[5];    // stage n+1: material multipliers of the 4 vapour species, energy
};

// Emitter concept:
//   static constexpr bool want_res, want_jac, want_hes;
//   void res(int r, double v); void jac(int r, int lv, double v); void hes(int i, int j, double v);
//
// FP64 instructions bound the evaluation on the device (one warp instruction per 19 cycles and
// SM), so the terms are arranged for few of them: products by structural zeros and ones are left
// out by hand (the compiler may not drop 0 x), Henry's second derivatives are formed per class of
// species instead of per pair, one division serves several reciprocals.  Every loop unrolls, so
// an emitter that keeps only some rows or entries leaves out what only the others need.  Every
// product that is added to something is an explicit fma or a rounded product (mul_rn), so a value
// comes out the same whatever else an instance computes.
#ifdef __CUDACC__
// ln(x) for the residuals and the barrier: x = 2^e m, m in [1, 2), from 1 / c rounded to 11 bits at the
// nearest c = 1 + j / 512, r = m / c - 1 (exact, |r| < 2^-9.6), ln x = e ln 2 + ln c + (r - r^2 / 2 + ... -
// r^6 / 6) (the table-driven method of Tang 1990).  From j = 213 on m / 2 and e + 1 are taken, so that x next
// to 1 has e = 0, c = 1 and no cancellation; ln 2 and ln c as a multiple of 2^-42 (their sum exact) and
// a rest.  12 FP64 instructions against about 30 of log(), within a unit in the last place as that.
// Anything but a positive normal number goes to log().
struct __align__(16) LnEntry {
    double hi, lo;   // -ln(1 / c) (of 2 / c from j = 213 on) in two parts; in hi's last 11 bits 2048 / c - 1024
};
constexpr int LN_TAB = 513, LN_HALF = 213;
__device__ LnEntry g_ln[LN_TAB];

inline void fill_ln_table(LnEntry* t) {
    for (int j = 0; j < LN_TAB; ++j) {
        const long double inv = roundl(2048.0L / (1.0L + (long double)j / 512)) / 2048;
        const long double v = -logl(j >= LN_HALF ? 2 * inv : inv);
        double hi = (double)(roundl(v * 0x1p42L) * 0x1p-42L);   // |hi| < 0.36: its last 12 bits are zero
        t[j].lo = (double)(v - (long double)hi);
        uint64_t bits;
        memcpy(&bits, &hi, sizeof(bits));
        bits |= (uint64_t)(inv * 2048) - 1024;
        memcpy(&t[j].hi, &bits, sizeof(bits));
    }
}
#endif
__host__ __device__ inline double ln_tab(double x) {
#ifdef __CUDA_ARCH__
    const int hi = __double2hiint(x);
    if (!(hi >= 0x00100000 && hi < 0x7ff00000)) return log(x);
    const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
    const int j = ((hi & 0x000fffff) + 0x400) >> 11;
    const LnEntry t = g_ln[j];
    const int code = __double2loint(t.hi);
    const double inv = __hiloint2double(0x3fe00000 + ((code & 0x7ff) << 10), 0);
    const double thi = __hiloint2double(__double2hiint(t.hi), code & ~0x7ff);
    const double e = (double)((hi >> 20) - 1023 + (j >= LN_HALF));
    const double r = fma(m, inv, -1.0);
    double q = fma(r, -1.0 / 6.0, 0.2);
    q = fma(r, q, -0.25);
    q = fma(r, q, 1.0 / 3.0);
    q = fma(r, q, -0.5);
    const double h = fma(e, 0x1.62e42fefa38p-1, thi), lo = fma(e, 0x1.ef35793c7673p-45, t.lo);   // ln 2 in two parts
    return h + (r + fma(r * r, q, lo));
#else
    return log(x);
#endif
}

// a b rounded, never contracted into a following sum
__host__ __device__ inline double mul_rn(double a, double b) {
#ifdef __CUDA_ARCH__
    return __dmul_rn(a, b);
#else
    return a * b;
#endif
}

#ifdef __CUDACC__
#pragma nv_exec_check_disable
#endif
template <class E>
__host__ __device__ inline void stage_eval(const Params& P, const StageIn& in, const StageLam* lam,
                                           E& e) {
    constexpr bool WR = E::want_res, WJ = E::want_jac, WH = E::want_hes;
    const double sT = P.sT;
    double x[9], y[4];
#pragma unroll
    for (int l = 0; l < 9; ++l) x[l] = mul_rn(P.sx[l], in.q[LX + l]);
#pragma unroll
    for (int j = 0; j < 4; ++j) y[j] = mul_rn(P.sy[j], in.q[LY + j]);
    const double L = in.q[LL], V = in.q[LV], T = mul_rn(sT, in.q[LT]);
    double xa[9], yb[4];
#pragma unroll
    for (int l = 0; l < 9; ++l) xa[l] = in.qa[l];
#pragma unroll
    for (int j = 0; j < 4; ++j) yb[j] = in.qb[j];
    const double La = in.qa[9], Ta = in.qa[10];
    const double Vb = in.qb[4], Tb = in.qb[5];
    const double Pr = in.P;

    // ---- reciprocals of T + C (Antoine), the stage pressure, the apparent-fraction total
    // of (9b) and T from one division: a = Tc Pr, b = tot T, r = 1 / (a b), then
    // 1/Tc = r b Pr, 1/Pr = r b Tc, 1/tot = r a T, 1/T = r a tot (all positive and O(1e-3
    // .. 1e3) at interior points)
    const double am = x[0] + x[1] + x[3];
    const double ac = x[3] + x[4] + x[6] + x[7];
    const double aw = x[4] + x[5] + x[6] + x[8];
    const double tot = am + ac + aw;
    const double Tc = T + P.psat_c;
    const double ra = Tc * Pr, rb = tot * T;
    const double r4 = 1.0 / (ra * rb);
    const double rbr = r4 * rb, rar = r4 * ra;
    const double iTc = rbr * Pr, iPr = rbr * Tc, it = rar * T, invT = rar * tot;

    // ---- enthalpies: h = h0 + dT (cpa + cpb / 2 dT), cp = cpa + cpb dT ----------------------
    const double dT = T - P.T_ref, dTa = Ta - P.T_ref, dTb = Tb - P.T_ref;
    const double hdT = 0.5 * dT, hdTa = 0.5 * dTa, hdTb = 0.5 * dTb;
    double hL[9], hV[4], hLa[9], hVb[4];
    double HL = 0, HV = 0, CL = 0, CV = 0, HLa = 0, HVb = 0, CLa = 0, CVb = 0;
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        hL[l] = fma(dT, fma(P.hL_cpb[l], hdT, P.hL_cpa[l]), P.hL0[l]);
        hLa[l] = fma(dTa, fma(P.hL_cpb[l], hdTa, P.hL_cpa[l]), P.hL0[l]);
        HL = fma(x[l], hL[l], HL);
        HLa = fma(xa[l], hLa[l], HLa);
        if (WJ || WH) CL = fma(x[l], fma(P.hL_cpb[l], dT, P.hL_cpa[l]), CL);
        if (WJ) CLa = fma(xa[l], fma(P.hL_cpb[l], dTa, P.hL_cpa[l]), CLa);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        hV[j] = fma(dT, fma(P.hV_cpb[j], hdT, P.hV_cpa[j]), P.hV0[j]);
        hVb[j] = fma(dTb, fma(P.hV_cpb[j], hdTb, P.hV_cpa[j]), P.hV0[j]);
        HV = fma(y[j], hV[j], HV);
        HVb = fma(yb[j], hVb[j], HVb);
        if (WJ || WH) CV = fma(y[j], fma(P.hV_cpb[j], dT, P.hV_cpa[j]), CV);
        if (WJ) CVb = fma(yb[j], fma(P.hV_cpb[j], dTb, P.hV_cpa[j]), CVb);
    }

    // ---- (9a) water saturation pressure ---------------------------------------------
    const double ps = exp(fma(-P.psat_b, iTc, P.psat_a));
    const double bT2 = P.psat_b * iTc * iTc;
    const double ps1 = ps * bT2;                                // dPsat/dT
    const double ps2 = ps * fma(bT2, bT2, -2.0 * bT2 * iTc);    // d2Psat/dT2
    // reciprocals of the scaled liquid fractions (derivatives of their logarithms), all
    // nine from one division: prefix products p_c = q_0 ... q_c, r = 1 / p_8, then walking
    // back 1/q_c = r p_{c-1} and r <- r q_c (the fractions are positive and O(1))
    double iq[9];
    if (WJ || WH) {
        double pre[9];
        pre[0] = in.q[LX];
#pragma unroll
        for (int c = 1; c < 9; ++c) pre[c] = pre[c - 1] * in.q[LX + c];
        double r = 1.0 / pre[8];
#pragma unroll
        for (int c = 8; c > 0; --c) {
            iq[c] = r * pre[c - 1];
            r *= in.q[LX + c];
        }
        iq[0] = r;
    } else {
#pragma unroll
        for (int c = 0; c < 9; ++c) iq[c] = 0.0;
    }

    // ---- (9b) Henry coefficient: ln H = ha + hb / T + s, s = hm x_MEA^app + hw x_H2O^app; for a
    // species of class c, ds/dx = (a_c - s t_c) / tot, a_c the class's hm, hw or 0 --------------
    const double sh = fma(P.henry_m, am * it, P.henry_w * (aw * it));
    const double Hh = exp(fma(P.henry_b, invT, P.henry_a) + sh);
    const double gT = -P.henry_b * invT * invT;
    double gc[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        const double a = cls_a(c) == 1 ? P.henry_m : (cls_a(c) == 2 ? P.henry_w : 0.0);
        const double ts = cls_t(c) == 2 ? 2.0 * sh : sh;
        gc[c] = cls_a(c) ? (a - ts) * it : -ts * it;
    }
    const double rhoH = P.rho_L * Hh;
    const double x7 = x[7];

    // ---- residuals ---------------------------------------------------------------------
    if (WR) {
#pragma unroll
        for (int c = 0; c < 11; ++c) {
            double r = 0.0;
            if (c < 9) r = fma(L, x[c], -La * xa[c]);
            if (c >= 7) {
                const double v = fma(V, y[c < 7 ? 0 : c - 7], -Vb * yb[c < 7 ? 0 : c - 7]);
                r = c < 9 ? r + v : v;
            }
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                if (nu(c, k) > 0) r -= in.q[LE + k];
                if (nu(c, k) < 0) r += in.q[LE + k];
            }
            e.res(c, r);
        }
        e.res(R_VH, fma(Pr, y[1], -x[8] * ps));
        e.res(R_VC, fma(Pr, y[0], -rhoH * x7));
        // sum_c nu_ck ln x_c as one logarithm per reaction: every nu is +-1, so it is
        // ln(prod over products of q_c / prod over reactants of q_c) + sum_c nu_ck ln sx_c
        // (the scaled fractions are O(1): the quotients stay far from over- and underflow)
        const double lT = ln_tab(T);
        // the five quotients' denominators inverted together from one division (prefix
        // products, then back)
        double qn[5], qd[5], pre[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            double num = 0.0, den = 0.0;
            bool hn = false, hd = false;
#pragma unroll
            for (int c = 0; c < 9; ++c) {
                if (nu(c, k) > 0) {
                    num = hn ? num * in.q[LX + c] : in.q[LX + c];
                    hn = true;
                }
                if (nu(c, k) < 0) {
                    den = hd ? den * in.q[LX + c] : in.q[LX + c];
                    hd = true;
                }
            }
            qn[k] = num;
            qd[k] = den;
            pre[k] = k ? pre[k ? k - 1 : 0] * den : den;
        }
        double rq = 1.0 / pre[4];
#pragma unroll
        for (int k = 4; k >= 0; --k) {
            const double rk = k ? rq * pre[k ? k - 1 : 0] : rq;
            if (k) rq *= qd[k];
            const double lnK = fma(P.KE_D[k], T, fma(P.KE_C[k], lT, fma(P.KE_B[k], invT, P.KE_A[k])));
            e.res(R_RX + k, (P.lnsxr[k] - lnK) + ln_tab(qn[k] * rk));
        }
        double sx_ = -1.0, sy_ = -1.0;
#pragma unroll
        for (int l = 0; l < 9; ++l) sx_ += x[l];
#pragma unroll
        for (int j = 0; j < 4; ++j) sy_ += y[j];
        e.res(R_SX, sx_);
        e.res(R_SY, sy_);
        e.res(R_E, fma(L, HL, -La * HLa) + fma(V, HV, -Vb * HVb));
        e.res(R_H, fma(V, P.R * T * iPr, fma(-0.25 * M_PI * P.u_max, in.d * in.d, in.q[LS])));
    }

    // ---- Jacobian ----------------------------------------------------------------------
    if (WJ) {
        const double nLa = -La, nVb = -Vb;
#pragma unroll
        for (int c = 0; c < 11; ++c) {
            if (c < 9) {
                const double f = L * P.sx[c];
                e.jac(c, LX + c, f);
                e.jac(c, LL, x[c]);
                e.jac(R_E, LX + c, f * hL[c]);
                if (in.has_above) {
                    const double fa = nLa * P.sx[c];
                    e.jac(c, AX + c, fa);
                    e.jac(c, AL, -xa[c]);
                    e.jac(R_E, AX + c, fa * hLa[c]);
                }
            }
            if (c >= 7) {
                const int j = c - 7;
                const double f = V * P.sy[j];
                e.jac(c, LY + j, f);
                e.jac(c, LV, y[j]);
                e.jac(R_E, LY + j, f * hV[j]);
                if (in.has_below) {
                    const double fb = nVb * P.sy[j];
                    e.jac(c, BY + j, fb);
                    e.jac(c, BV, -yb[j]);
                    e.jac(R_E, BY + j, fb * hVb[j]);
                }
            }
#pragma unroll
            for (int k = 0; k < 5; ++k)
                if (nu(c, k) != 0) e.jac(c, LE + k, -(double)nu(c, k));
        }
        // (9a)
        e.jac(R_VH, LY + 1, Pr * P.sy[1]);
        e.jac(R_VH, LX + 8, -P.sx[8] * ps);
        e.jac(R_VH, LT, -x[8] * ps1 * sT);
        // (9b)
        const double rx7 = -rhoH * x7;
        e.jac(R_VC, LY + 0, Pr * P.sy[0]);
        double vc[5];
#pragma unroll
        for (int c = 0; c < 5; ++c) vc[c] = c == 4 ? fma(rx7, gc[c], -rhoH) : rx7 * gc[c];
#pragma unroll
        for (int k = 0; k < 9; ++k)
            if (in_henry(k)) e.jac(R_VC, LX + k, vc[henry_cls(k) < 0 ? 0 : henry_cls(k)] * P.sx[k]);
        e.jac(R_VC, LT, rx7 * gT * sT);
        // (3a)
        const double sTi = sT * invT;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
#pragma unroll
            for (int c = 0; c < 9; ++c)
                if (nu(c, k) != 0) e.jac(R_RX + k, LX + c, nu(c, k) > 0 ? iq[c] : -iq[c]);
            e.jac(R_RX + k, LT, fma(sTi, fma(P.KE_B[k], invT, -P.KE_C[k]), -sT * P.KE_D[k]));
        }
        // (4)
#pragma unroll
        for (int l = 0; l < 9; ++l) e.jac(R_SX, LX + l, P.sx[l]);
#pragma unroll
        for (int j = 0; j < 4; ++j) e.jac(R_SY, LY + j, P.sy[j]);
        // (6)
        e.jac(R_E, LL, HL);
        e.jac(R_E, LV, HV);
        e.jac(R_E, LT, sT * fma(L, CL, V * CV));
        if (in.has_above) {
            e.jac(R_E, AL, -HLa);
            e.jac(R_E, AT, sT * nLa * CLa);
        }
        if (in.has_below) {
            e.jac(R_E, BV, -HVb);
            e.jac(R_E, BT, sT * nVb * CVb);
        }
        // (10b)
        e.jac(R_H, LV, P.R * T * iPr);
        e.jac(R_H, LT, V * (P.R * sT) * iPr);
        e.jac(R_H, LS, 1.0);
        e.jac(R_H, LD_, (-0.5 * M_PI * P.u_max) * in.d);
    }

    // ---- Lagrangian Hessian block of this stage's unknowns (lower triangle) ------------
    // Terms come from this stage's rows and from the neighbours' rows in which this
    // stage's streams appear: the stage below reads (L, x, T) of this stage as its
    // "from above" stream, the stage above reads (V, y, T) as its "from below" stream.
    if (WH) {
        const double* lo = lam->own;
        double muL[9], muV[4];
#pragma unroll
        for (int c = 0; c < 9; ++c) muL[c] = in.has_below ? lo[c] - lam->below[c] : lo[c];
#pragma unroll
        for (int j = 0; j < 4; ++j) muV[j] = in.has_above ? lo[7 + j] - lam->above[j] : lo[7 + j];
        const double muEL = in.has_below ? lo[R_E] - lam->below[9] : lo[R_E];
        const double muEV = in.has_above ? lo[R_E] - lam->above[4] : lo[R_E];
        const double lVH = lo[R_VH], lVC = lo[R_VC], lH = lo[R_H];

        // Henry block over the species of the apparent totals (and the ln x diagonals).  With g_k =
        // (a_k - s t_k) / tot the second derivatives of H x7 / (H x7) are g_k g_l + dg_k/dx_l =
        // ((a_k - p t_k)(a_l - p t_l) - t_k t_l) / tot^2, p = 1 + s: one value per pair of classes
        const double c0 = -lVC * rhoH;
        const double c7 = c0 * x7 * it * it, p1 = 1.0 + sh;
        double bc[5], pc[15], g0[5];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            const double a = cls_a(c) == 1 ? P.henry_m : (cls_a(c) == 2 ? P.henry_w : 0.0);
            const double tp = cls_t(c) == 2 ? 2.0 * p1 : p1;
            bc[c] = cls_a(c) ? a - tp : -tp;
            g0[c] = mul_rn(c0, gc[c]);
        }
#pragma unroll
        for (int c = 0; c < 5; ++c)
#pragma unroll
            for (int d = 0; d <= c; ++d) {
                double v = mul_rn(c7, fma(bc[c], bc[d], -(double)(cls_t(c) * cls_t(d))));
                if (c == 4) v += d == 4 ? 2.0 * g0[4] : g0[d];   // the factor x7 itself
                pc[c * (c + 1) / 2 + d] = v;
            }
#pragma unroll
        for (int k = 0; k < 9; ++k) {
#pragma unroll
            for (int l = 0; l <= k; ++l) {
                const bool henry = in_henry(k) && in_henry(l);
                double a = 0.0;
                bool any = false;
                if (k == l) {
#pragma unroll
                    for (int r = 0; r < 5; ++r) {
                        if (nu(k, r) > 0) a = any ? a + lo[R_RX + r] : lo[R_RX + r];
                        if (nu(k, r) < 0) a = any ? a - lo[R_RX + r] : -lo[R_RX + r];
                        any = any || nu(k, r) != 0;
                    }
                }
                if (!henry && !any) continue;
                double v = any ? -a * (iq[k] * iq[k]) : 0.0;
                if (henry) {
                    const int ck = henry_cls(k) < 0 ? 0 : henry_cls(k), cl = henry_cls(l) < 0 ? 0 : henry_cls(l);
                    const int hi = ck > cl ? ck : cl, lw = ck > cl ? cl : ck;
                    const double q = pc[hi * (hi + 1) / 2 + lw], w = P.sxx[k * (k + 1) / 2 + l];
                    v = any ? fma(q, w, v) : q * w;
                }
                e.hes(LX + k, LX + l, v);
            }
        }
        // (L, x_l) and (V, y_j): bilinear flows in (1) and (6)
#pragma unroll
        for (int l = 0; l < 9; ++l) e.hes(LL, LX + l, P.sx[l] * fma(muEL, hL[l], muL[l]));
#pragma unroll
        for (int j = 0; j < 4; ++j) e.hes(LV, LY + j, P.sy[j] * fma(muEV, hV[j], muV[j]));
        // (T, x_l)
        const double aL = sT * muEL * L, aV = sT * muEV * V;
        const double hT = c0 * gT * sT, hT7 = hT * x7;
        double tc[5];
#pragma unroll
        for (int c = 0; c < 5; ++c) tc[c] = c == 4 ? fma(hT7, gc[c], hT) : hT7 * gc[c];
#pragma unroll
        for (int l = 0; l < 9; ++l) {
            const double cp = fma(P.hL_cpb[l], dT, P.hL_cpa[l]);
            double v = in_henry(l) ? fma(aL, cp, tc[henry_cls(l) < 0 ? 0 : henry_cls(l)]) : aL * cp;
            if (l == 8) v = fma(-lVH * sT, ps1, v);
            e.hes(LT, LX + l, v * P.sx[l]);
        }
        // (T, y_j)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            e.hes(LT, LY + j, aV * fma(P.hV_cpb[j], dT, P.hV_cpa[j]) * P.sy[j]);
        e.hes(LT, LL, sT * muEL * CL);
        e.hes(LT, LV, sT * fma(muEV, CV, lH * P.R * iPr));
        // (T, T)
        {
            double dCL = 0.0, dCV = 0.0, rx = 0.0;
#pragma unroll
            for (int l = 0; l < 9; ++l) dCL = fma(x[l], P.hL_cpb[l], dCL);
#pragma unroll
            for (int j = 0; j < 4; ++j) dCV = fma(y[j], P.hV_cpb[j], dCV);
            const double i2 = invT * invT, ti = 2.0 * invT;
#pragma unroll
            for (int r = 0; r < 5; ++r) rx = fma(lo[R_RX + r], fma(P.KE_B[r], ti, -P.KE_C[r]), rx);
            double v = fma(muEL * L, dCL, muEV * V * dCV);
            v = fma(-lVH * x[8], ps2, v);
            v = fma(c0 * x7, fma(gT, gT, 2.0 * P.henry_b * i2 * invT), v);
            v = fma(-i2, rx, v);
            e.hes(LT, LT, sT * sT * v);
        }
    }
}

}  // namespace absorber
