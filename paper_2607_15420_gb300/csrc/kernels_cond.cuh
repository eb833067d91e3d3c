// kernels_cond.cuh -- the scenario blocks J_s factored and solved through condensed stage
// systems (A4-A6), in FP64 or FP32, and the fused Newton-direction kernels built on them.
//
// A stage's 22 unknowns and rows condense by fixed pivots to a core of 7:
//   * the extents: each of R1, R2, R3, R4, R5 alone enters one material row (MEAH+, CO3--,
//     OH-, MEACOO-, CO2) with coefficient +-1, so those rows give the extents, and the
//     rows of MEA, H+, HCO3-, H2O combined with them balance moieties without extents;
//   * the slack: coefficient 1 in the hydraulic row, which nothing else needs;
//   * H+, HCO3-, OH-, CO3--, CO2 from the equilibria R1, R4, R3, R2, R5 in that order (their
//     coefficients are +-1 / x: in relative fractions the pivots are 1, the largest entries
//     of their columns), H2O from sum x, the vapour fractions of H2O, CO2, N2 from (9a),
//     (9b) and sum y (pivots P, P and 1).
// The multipliers of all these pivots are of order one (at most 7 over iterates of whole
// solves), so the order is as safe as partial pivoting, and what is left -- unknowns x_MEA,
// x_MEAH+, x_MEACOO-, T, L, V, y_O2; rows a (MEA), b, c, d (moieties), N, O (N2, O2),
// E (energy) -- has condition 1e3..1e4.  Neighbouring stages meet in five quantities only,
// the vapour's g = N u (CO2, H2O, N2, O2 flows, enthalpy) and the liquid's l = M u (four
// moiety flows, enthalpy):
//     A u_n - E' g_{n-1} - E l_{n+1} = r_n,
// with E the rows a, b, c, d, E and E' the rows (b + c - d), d, N, O, E.  The block LU over
// stages is At_n = A_n - E' K_{n-1} M_n, K_n = N_n At_n^-1 E.  The factorization stores each
// At_n^-1 (7 x 7, Gauss-Jordan with partial pivoting) and the 5 x 5 maps D_n = N At^-1 E',
// T_n = M At^-1 E, so a solve is: every stage's products at once, a chain of nine 5 x 5
// products up the column (g_n = ghat_n + D_n g_{n-1}), every stage, a chain down
// (l_n = lhat_n + T_n l_{n+1}), every stage.  J^T is solved with the same data transposed.
//
// Against a block LU over the 22 x 22 stage blocks this takes about 1,000 instead of 8,300
// fused multiply-adds per stage of a factorization and 250 instead of 740 of a solve, and
// 2 KB (FP64) instead of 5.8 KB of factors per stage.  Its errors against extended precision, over
// iterates of whole solves, are those of the block LU to within a factor of 1.6 either way
// (geometric means, FP64 and FP32).
//
// FP64 issues at one warp instruction per 19 cycles and SM (64 cycles on one of its four
// schedulers), so FP64 instructions bound the kernels in FP64, and the chains' latency the
// small sizes and FP32.
//
// The Jacobian values are those of the evaluation: the extents' coefficients -nu, the
// slack's 1, and a stage's stream entries in its neighbours' rows the negatives of its own.  A
// Jacobian from outside the library is checked for that (condense_conforms); where it differs
// the 22 x 22 stage blocks are factored as they are (kernels_warp.cuh).
#pragma once

#include "kernels.cuh"
#include "vec_kernels.cuh"

namespace absorber {

constexpr int NCORE = 7;   // core unknowns: x0, x1, x3, T, L, V, y3; rows a, b, c, d, N, O, E
constexpr int NLINK = 5;   // quantities between neighbouring stages, each way

// stored values of a stage (entry e of stage n, scenario s at F[(n NF + e) ld + s]).  x2 x4 x5
// x6 x7 x8, y1 y0 y2: the eliminated fractions, in elimination order
enum CondField {
    CF_I12 = 0, CF_I44, CF_I35, CF_I26, CF_I57, CF_I8, CF_IY1, CF_IY0, CF_IY2,   // reciprocal pivots
    CF_A32 = 9, CF_A24, CF_A22, CF_A52, CF_A54,         // equilibrium rows over their pivots
    CF_C2 = 14, CF_C4, CF_C5, CF_C6, CF_C7,             // sum x over the pivot of x8
    CF_X48 = 19, CF_X58, CF_X68, CF_X78,                // x4..x7 per x8 before its elimination
    CF_H18 = 23,                                        // (9a): x8 over the pivot
    CF_K4 = 24,                                         // (9b): x4..x8 over the pivot
    CF_D0 = 29, CF_D1 = 30,                             // sum y: y0, y1 over the pivot
    CF_MC = 31,                                         // material rows 1..8: own fraction
    CF_W0 = 39, CF_W1, CF_W2,                           // material rows of CO2, H2O, N2: own y
    CF_H2 = 42, CF_H4, CF_H5, CF_H6, CF_H7, CF_H8,      // energy row: x2, x4..x8
    CF_Z0 = 48,                                         // energy row: y0, y1, y2
    CF_X = 51,                                          // x2 by (x0, x1, T); x4..x8 by (x0, x1, x3, T)
    CF_Y0 = 74, CF_Y1 = 78, CF_Y2 = 82, CF_Y23 = 86,    // y0, y1, y2 by (x0, x1, x3, T); y2 by y3
    CF_L1 = 87, CF_L3, CF_L5, CF_L6, CF_L7,             // material rows: L
    CF_VV = 92,                                         // material row of CO2: V
    CF_HV = 93, CF_HT = 94,                             // hydraulic row: V, T
    CF_M = 95,                                          // l by (x0, x1, x3, T, L), 5 x 5
    CF_N = 120,                                         // g by (x0, x1, x3, T, V, y3), 5 x 6
    CF_INV = 150,                                       // At^-1, 7 x 7
    CF_D = 199, CF_T = 224,                             // 5 x 5 link maps
    CF_COUNT = 249
};

// structural zeros of M (row a does not see T) and N (O2 sees V, y3 only; CO2, H2O no y3)
__host__ __device__ constexpr bool m_has(int i, int j) { return !(i == 0 && j == 3); }
__host__ __device__ constexpr bool n_has(int i, int j) { return i == 3 ? j >= 4 : (j < 5 || i == 2 || i == 4); }
// core unknown behind column j of N
__host__ __device__ constexpr int n_core(int j) { return j < 4 ? j : (j == 4 ? 5 : 6); }
// core row behind liquid link k (a, b, c, d, E)
__host__ __device__ constexpr int e_row(int k) { return k < 4 ? k : 6; }

template <class T>
struct CondRef {   // the stored values of one stage of one scenario
    T* f;
    int64_t ld;
    __device__ T& operator()(int e) const { return f[(int64_t)e * ld]; }
};
template <class T>
__device__ inline CondRef<T> cond_ref(T* F, int64_t ld, int n, int64_t s) {
    return CondRef<T>{F + (int64_t)n * CF_COUNT * ld + s, ld};
}

// 1 / a: the hardware's approximate reciprocal and one step of the hyperpower iteration (Altman 1960),
// e = 1 - a r: of third order r (1 + e + e^2) for FP64 (three dependent FP64 operations, against five of a
// pair of second order), of second for FP32; within a unit in the last place for |a| in 2^-1000 .. 2^1000
// and 2^-124 .. 2^124, as a division; beyond that (the hardware's takes subnormal numbers as 0) not
__device__ inline double cond_recip(double a) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
    const double e = fma(-a, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
__device__ inline float cond_recip(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return fmaf(r, fmaf(-a, r, 1.0f), r);
}
__device__ inline double cond_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ inline float cond_fma(float a, float b, float c) { return fmaf(a, b, c); }

// |a| <= lim, false for NaN
__device__ __forceinline__ bool within(double a, double lim) {
    return mag_key(a) <= (unsigned long long)__double_as_longlong(lim);
}
__device__ __forceinline__ bool within(float a, float lim) { return fabsf(a) <= lim; }

// Condense one stage: A(r, lv) its own Jacobian entries, Lt the energy row's liquid share of
// dT, Vt its vapour share (Lt + Vt = A(R_E, LT)); into f, all but At^-1, D, T.  True where the
// fixed pivots are safe: x_H2O's, a sum of terms of one sign at interior points, is no less than
// 1 / 256 of any term, the others are finite.
template <class T, class Own>
__device__ inline bool condense_stage(const Own& A, T Lt, T Vt, const CondRef<T>& f) {
    // ---- equilibria: x2 (R1), x4 (R4), x5 (R3), x6 (R2), x7 (R5) -----------------------------
    constexpr int R1 = R_RX, R2 = R_RX + 1, R3 = R_RX + 2, R4 = R_RX + 3, R5 = R_RX + 4;
    const T i12 = cond_recip(A(R1, 2)), i44 = cond_recip(A(R4, 4)), i35 = cond_recip(A(R3, 5)),
            i26 = cond_recip(A(R2, 6)), i57 = cond_recip(A(R5, 7));
    const T a32 = A(R3, 2) * i35, a24 = A(R2, 4) * i26, a22 = A(R2, 2) * i26, a52 = A(R5, 2) * i57,
            a54 = A(R5, 4) * i57;
    // rows of coefficients on (x0, x1, x3, T), and on x8 while it is still there
    T X2[4], X4[4], X5[4], X6[4], X7[4], X8[4];
    X2[0] = -A(R1, 0) * i12;
    X2[1] = -A(R1, 1) * i12;
    X2[2] = T(0);
    X2[3] = -A(R1, LT) * i12;
    X4[0] = -A(R4, 0) * i44;
    X4[1] = T(0);
    X4[2] = -A(R4, 3) * i44;
    X4[3] = -A(R4, LT) * i44;
    const T X48 = -A(R4, 8) * i44, X58 = -A(R3, 8) * i35;
    X5[0] = -a32 * X2[0];
    X5[1] = -a32 * X2[1];
    X5[2] = T(0);
    X5[3] = cond_fma(-a32, X2[3], -A(R3, LT) * i35);
    X6[0] = cond_fma(-a24, X4[0], -a22 * X2[0]);
    X6[1] = -a22 * X2[1];
    X6[2] = -a24 * X4[2];
    X6[3] = cond_fma(-a24, X4[3], cond_fma(-a22, X2[3], -A(R2, LT) * i26));
    const T X68 = -a24 * X48;
    X7[0] = cond_fma(-a52, X2[0], -a54 * X4[0]);
    X7[1] = -a52 * X2[1];
    X7[2] = -a54 * X4[2];
    X7[3] = cond_fma(-a52, X2[3], cond_fma(-a54, X4[3], -A(R5, LT) * i57));
    const T X78 = cond_fma(-a54, X48, -A(R5, 8) * i57);
    f(CF_I12) = i12;
    f(CF_I44) = i44;
    f(CF_I35) = i35;
    f(CF_I26) = i26;
    f(CF_I57) = i57;
    f(CF_A32) = a32;
    f(CF_A24) = a24;
    f(CF_A22) = a22;
    f(CF_A52) = a52;
    f(CF_A54) = a54;
    f(CF_X48) = X48;
    f(CF_X58) = X58;
    f(CF_X68) = X68;
    f(CF_X78) = X78;
    // ---- sum x: x8 -----------------------------------------------------------------------------
    const T c2 = A(R_SX, 2), c4 = A(R_SX, 4), c5 = A(R_SX, 5), c6 = A(R_SX, 6), c7 = A(R_SX, 7);
    const T i8 = cond_recip(cond_fma(c4, X48, cond_fma(c5, X58, cond_fma(c6, X68, cond_fma(c7, X78, (T)A(R_SX, 8))))));
    const T s2 = c2 * i8, s4 = c4 * i8, s5 = c5 * i8, s6 = c6 * i8, s7 = c7 * i8;
    const T c013[4] = {(T)A(R_SX, 0), (T)A(R_SX, 1), (T)A(R_SX, 3), T(0)};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        T a = q < 3 ? c013[q] * i8 : T(0);
        if (q != 2) a = cond_fma(s2, X2[q], a);
        if (q != 1) a = cond_fma(s4, X4[q], a);
        if (q != 2) a = cond_fma(s5, X5[q], a);
        a = cond_fma(s6, X6[q], a);
        a = cond_fma(s7, X7[q], a);
        X8[q] = -a;
        X4[q] = cond_fma(X48, X8[q], X4[q]);
        X5[q] = cond_fma(X58, X8[q], X5[q]);
        X6[q] = cond_fma(X68, X8[q], X6[q]);
        X7[q] = cond_fma(X78, X8[q], X7[q]);
    }
    f(CF_I8) = i8;
    f(CF_C2) = s2;
    f(CF_C4) = s4;
    f(CF_C5) = s5;
    f(CF_C6) = s6;
    f(CF_C7) = s7;
    f(CF_X + 0) = X2[0];
    f(CF_X + 1) = X2[1];
    f(CF_X + 2) = X2[3];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        f(CF_X + 3 + q) = X4[q];
        f(CF_X + 7 + q) = X5[q];
        f(CF_X + 11 + q) = X6[q];
        f(CF_X + 15 + q) = X7[q];
        f(CF_X + 19 + q) = X8[q];
    }
    // ---- vapour fractions: y1 (9a), y0 (9b), y2 (sum y) -----------------------------------------
    const T iy1 = cond_recip(A(R_VH, LY + 1)), iy0 = cond_recip(A(R_VC, LY)), iy2 = cond_recip(A(R_SY, LY + 2));
    const T h18 = A(R_VH, 8) * iy1;
    const T k4 = A(R_VC, 4) * iy0, k5 = A(R_VC, 5) * iy0, k6 = A(R_VC, 6) * iy0, k7 = A(R_VC, 7) * iy0,
            k8 = A(R_VC, 8) * iy0;
    const T d0 = A(R_SY, LY) * iy2, d1 = A(R_SY, LY + 1) * iy2, y23 = -A(R_SY, LY + 3) * iy2;
    const T kq[4] = {(T)A(R_VC, 0), (T)A(R_VC, 1), (T)A(R_VC, 3), (T)A(R_VC, LT)};
    T Y0[4], Y1[4], Y2[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        Y1[q] = -h18 * X8[q];
        if (q == 3) Y1[q] = cond_fma(-(T)A(R_VH, LT), iy1, Y1[q]);
        T a = kq[q] * iy0;
        a = cond_fma(k4, X4[q], a);
        a = cond_fma(k5, X5[q], a);
        a = cond_fma(k6, X6[q], a);
        a = cond_fma(k7, X7[q], a);
        a = cond_fma(k8, X8[q], a);
        Y0[q] = -a;
        Y2[q] = cond_fma(-d0, Y0[q], -d1 * Y1[q]);
        f(CF_Y0 + q) = Y0[q];
        f(CF_Y1 + q) = Y1[q];
        f(CF_Y2 + q) = Y2[q];
    }
    f(CF_Y23) = y23;
    f(CF_IY1) = iy1;
    f(CF_IY0) = iy0;
    f(CF_IY2) = iy2;
    f(CF_H18) = h18;
    f(CF_K4 + 0) = k4;
    f(CF_K4 + 1) = k5;
    f(CF_K4 + 2) = k6;
    f(CF_K4 + 3) = k7;
    f(CF_K4 + 4) = k8;
    f(CF_D0) = d0;
    f(CF_D1) = d1;
    // ---- liquid links M ---------------------------------------------------------------------------
    const T m0 = A(0, 0), m1 = A(1, 1), m2 = A(2, 2), m3 = A(3, 3), m4 = A(4, 4), m5 = A(5, 5), m6 = A(6, 6),
            m7 = A(7, 7), m8 = A(8, 8);
    const T l0 = A(0, LL), l1 = A(1, LL), l2 = A(2, LL), l3 = A(3, LL), l4 = A(4, LL), l5 = A(5, LL), l6 = A(6, LL),
            l7 = A(7, LL), l8 = A(8, LL);
    const T h2 = A(R_E, 2), h4 = A(R_E, 4), h5 = A(R_E, 5), h6 = A(R_E, 6), h7 = A(R_E, 7), h8 = A(R_E, 8);
    const T hq[4] = {(T)A(R_E, 0), (T)A(R_E, 1), (T)A(R_E, 3), Lt};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const T f5 = m5 * X5[q], f6 = m6 * X6[q], f7 = m7 * X7[q];
        f(CF_M + q) = q == 0 ? m0 : (q == 1 ? m1 : (q == 2 ? m3 : T(0)));
        f(CF_M + 5 + q) = cond_fma(m2, X2[q], (f7 - f6) - f5) + (q == 1 ? m1 : T(0));
        f(CF_M + 10 + q) = cond_fma(m4, X4[q], f6 + f7) + (q == 2 ? m3 : T(0));
        f(CF_M + 15 + q) = cond_fma(m8, X8[q], f5 - f7) - (q == 2 ? m3 : T(0));
        T a = hq[q];
        if (q != 2) a = cond_fma(h2, X2[q], a);
        a = cond_fma(h4, X4[q], a);
        a = cond_fma(h5, X5[q], a);
        a = cond_fma(h6, X6[q], a);
        a = cond_fma(h7, X7[q], a);
        f(CF_M + 20 + q) = cond_fma(h8, X8[q], a);
    }
    f(CF_M + 4) = l0 + l1 + l3;
    f(CF_M + 9) = ((l2 + l1) - (l6 + l5)) + l7;
    f(CF_M + 14) = (l4 + l6) + (l3 + l7);
    f(CF_M + 19) = (l8 + l5) - (l3 + l7);
    f(CF_M + 24) = A(R_E, LL);
    f(CF_MC + 0) = m1;
    f(CF_MC + 1) = m2;
    f(CF_MC + 2) = m3;
    f(CF_MC + 3) = m4;
    f(CF_MC + 4) = m5;
    f(CF_MC + 5) = m6;
    f(CF_MC + 6) = m7;
    f(CF_MC + 7) = m8;
    f(CF_L1) = l1;
    f(CF_L3) = l3;
    f(CF_L5) = l5;
    f(CF_L6) = l6;
    f(CF_L7) = l7;
    f(CF_H2) = h2;
    f(CF_H4) = h4;
    f(CF_H5) = h5;
    f(CF_H6) = h6;
    f(CF_H7) = h7;
    f(CF_H8) = h8;
    // ---- vapour links N -----------------------------------------------------------------------------
    const T w0 = A(7, LY), w1 = A(8, LY + 1), w2 = A(9, LY + 2), vv = A(7, LV);
    const T z0 = A(R_E, LY), z1 = A(R_E, LY + 1), z2 = A(R_E, LY + 2);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        f(CF_N + q) = w0 * Y0[q];
        f(CF_N + 6 + q) = w1 * Y1[q];
        f(CF_N + 12 + q) = w2 * Y2[q];
        f(CF_N + 18 + q) = T(0);
        f(CF_N + 24 + q) = cond_fma(z0, Y0[q], cond_fma(z1, Y1[q], z2 * Y2[q])) + (q == 3 ? Vt : T(0));
    }
    f(CF_N + 4) = vv;
    f(CF_N + 5) = T(0);
    f(CF_N + 10) = A(8, LV);
    f(CF_N + 11) = T(0);
    f(CF_N + 16) = A(9, LV);
    f(CF_N + 17) = w2 * y23;
    f(CF_N + 22) = A(10, LV);
    f(CF_N + 23) = A(10, LY + 3);
    f(CF_N + 28) = A(R_E, LV);
    f(CF_N + 29) = cond_fma(z2, y23, (T)A(R_E, LY + 3));
    f(CF_W0) = w0;
    f(CF_W1) = w1;
    f(CF_W2) = w2;
    f(CF_Z0 + 0) = z0;
    f(CF_Z0 + 1) = z1;
    f(CF_Z0 + 2) = z2;
    f(CF_VV) = vv;
    f(CF_HV) = A(R_H, LV);
    f(CF_HT) = A(R_H, LT);
    constexpr T TOP = sizeof(T) == 8 ? T(1.7976931348623157e308) : T(3.4028234663852886e38);   // finite
    return (int)within(i12, TOP) & within(iy1, TOP) & within(iy0, TOP) & within(iy2, TOP) &
           within((T)A(R_SX, 8) * i8, T(256)) & within(s4 * X48, T(256)) & within(s5 * X58, T(256)) &
           within(s6 * X68, T(256)) & within(s7 * X78, T(256));
}

// The right-hand side of the core: r -> rc; the eliminated fractions' own parts -> rho
// (x2, x4, x5, x6, x7, x8, y1, y0, y2), for cond_expand, and the flows they carry into the
// neighbours' core rows: lo (liquid, rows b, c, d, E of the stage below) and go (vapour: CO2,
// H2O, N2, enthalpy, of the stage above), which those stages add to their rc.
template <class T>
__device__ inline void cond_reduce(const CondRef<const T>& f, const T (&r)[NR], T (&rc)[NCORE], T (&rho)[9],
                                            T (&lo)[4], T (&go)[4]) {
    const T p2 = r[R_RX] * f(CF_I12);
    T p4 = r[R_RX + 3] * f(CF_I44);
    T p5 = cond_fma(-f(CF_A32), p2, r[R_RX + 2] * f(CF_I35));
    T p6 = cond_fma(-f(CF_A24), p4, cond_fma(-f(CF_A22), p2, r[R_RX + 1] * f(CF_I26)));
    T p7 = cond_fma(-f(CF_A52), p2, cond_fma(-f(CF_A54), p4, r[R_RX + 4] * f(CF_I57)));
    T p8 = cond_fma(-f(CF_C2), p2, r[R_SX] * f(CF_I8));
    p8 = cond_fma(-f(CF_C4), p4, p8);
    p8 = cond_fma(-f(CF_C5), p5, p8);
    p8 = cond_fma(-f(CF_C6), p6, p8);
    p8 = cond_fma(-f(CF_C7), p7, p8);
    p4 = cond_fma(f(CF_X48), p8, p4);
    p5 = cond_fma(f(CF_X58), p8, p5);
    p6 = cond_fma(f(CF_X68), p8, p6);
    p7 = cond_fma(f(CF_X78), p8, p7);
    const T y1 = cond_fma(-f(CF_H18), p8, r[R_VH] * f(CF_IY1));
    T y0 = r[R_VC] * f(CF_IY0);
    y0 = cond_fma(-f(CF_K4 + 0), p4, y0);
    y0 = cond_fma(-f(CF_K4 + 1), p5, y0);
    y0 = cond_fma(-f(CF_K4 + 2), p6, y0);
    y0 = cond_fma(-f(CF_K4 + 3), p7, y0);
    y0 = cond_fma(-f(CF_K4 + 4), p8, y0);
    const T y2 = cond_fma(-f(CF_D0), y0, cond_fma(-f(CF_D1), y1, r[R_SY] * f(CF_IY2)));
    const T f5 = f(CF_MC + 4) * p5, f6 = f(CF_MC + 5) * p6, f7 = f(CF_MC + 6) * p7;
    lo[0] = cond_fma(f(CF_MC + 1), p2, (f7 - f6) - f5);
    lo[1] = cond_fma(f(CF_MC + 3), p4, f6 + f7);
    lo[2] = cond_fma(f(CF_MC + 7), p8, f5 - f7);
    T e = f(CF_H2) * p2;
    e = cond_fma(f(CF_H4), p4, e);
    e = cond_fma(f(CF_H5), p5, e);
    e = cond_fma(f(CF_H6), p6, e);
    e = cond_fma(f(CF_H7), p7, e);
    lo[3] = cond_fma(f(CF_H8), p8, e);
    go[0] = f(CF_W0) * y0;
    go[1] = f(CF_W1) * y1;
    go[2] = f(CF_W2) * y2;
    go[3] = cond_fma(f(CF_Z0 + 0), y0, cond_fma(f(CF_Z0 + 1), y1, f(CF_Z0 + 2) * y2));
    const T r56 = r[5] + r[6], r37 = r[3] + r[7];
    rc[0] = r[0] + (r[1] + r[3]);
    rc[1] = ((r[2] + r[1]) - (r56 - r[7])) - (lo[0] + go[0]);
    rc[2] = ((r[4] + r[6]) + r37) - (lo[1] + go[0]);
    rc[3] = ((r[8] + r[5]) - r37) - (lo[2] + (go[1] - go[0]));
    rc[4] = r[9] - go[2];
    rc[5] = r[10];
    rc[6] = r[R_E] - (lo[3] + go[3]);
    rho[0] = p2;
    rho[1] = p4;
    rho[2] = p5;
    rho[3] = p6;
    rho[4] = p7;
    rho[5] = p8;
    rho[6] = y1;
    rho[7] = y0;
    rho[8] = y2;
}

// From the core unknowns c: the stage's fractions, flows and temperature into u, and the flows
// the extents need: fl = (f1, f3, f5, f6, f7: liquid flows of rows 1, 3, 5, 6, 7; CO2 vapour).
template <class T>
__device__ inline void cond_expand(const CondRef<const T>& f, const T (&c)[NCORE], const T (&rho)[9],
                                            T (&u)[NV], T (&fl)[6]) {
    u[0] = c[0];
    u[1] = c[1];
    u[3] = c[2];
    u[LT] = c[3];
    u[LL] = c[4];
    u[LV] = c[5];
    u[LY + 3] = c[6];
    u[2] = cond_fma(f(CF_X + 0), c[0], cond_fma(f(CF_X + 1), c[1], cond_fma(f(CF_X + 2), c[3], rho[0])));
#pragma unroll
    for (int k = 0; k < 5; ++k) {   // x4..x8
        T a = rho[1 + k];
#pragma unroll
        for (int q = 0; q < 4; ++q) a = cond_fma(f(CF_X + 3 + 4 * k + q), c[q], a);
        u[4 + k] = a;
    }
    T y0 = rho[7], y1 = rho[6], y2 = cond_fma(f(CF_Y23), c[6], rho[8]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        y0 = cond_fma(f(CF_Y0 + q), c[q], y0);
        y1 = cond_fma(f(CF_Y1 + q), c[q], y1);
        y2 = cond_fma(f(CF_Y2 + q), c[q], y2);
    }
    u[LY] = y0;
    u[LY + 1] = y1;
    u[LY + 2] = y2;
    fl[0] = cond_fma(f(CF_MC + 0), u[1], f(CF_L1) * c[4]);
    fl[1] = cond_fma(f(CF_MC + 2), u[3], f(CF_L3) * c[4]);
    fl[2] = cond_fma(f(CF_MC + 4), u[5], f(CF_L5) * c[4]);
    fl[3] = cond_fma(f(CF_MC + 5), u[6], f(CF_L6) * c[4]);
    fl[4] = cond_fma(f(CF_MC + 6), u[7], f(CF_L7) * c[4]);
    fl[5] = cond_fma(f(CF_W0), y0, f(CF_VV) * c[5]);
}

// The extents and the slack, from the stage's flows fl, the liquid flows of the stage above
// fa (zero for the top stage) and the CO2 vapour flow of the stage below vb (zero for the bottom).
template <class T>
__device__ inline void cond_extents(const CondRef<const T>& f, const T (&r)[NR], const T (&fl)[6],
                                             const T (&fa)[5], T vb, T (&u)[NV]) {
    u[LE + 0] = r[1] - (fl[0] - fa[0]);
    u[LE + 1] = (fl[3] - fa[3]) - r[6];
    u[LE + 2] = (fl[2] - fa[2]) - r[5];
    u[LE + 3] = r[3] - (fl[1] - fa[1]);
    u[LE + 4] = r[7] - ((fl[4] - fa[4]) + (fl[5] - vb));
    u[LS] = cond_fma(-f(CF_HV), u[LV], cond_fma(-f(CF_HT), u[LT], r[R_H]));
}

// J^T: the transpose of cond_expand / cond_extents.  g: the stage's gradient; ea, eb: the
// extents' entries of g of the stage above and below (zero past the ends).  Core right-hand
// side -> gc, the eliminated fractions' entries -> gam (x2, x4, x5, x6, x7, x8, y1, y0, y2).
template <class T>
__device__ inline void cond_reduce_t(const CondRef<const T>& f, const T (&g)[NV], T ea4, const T (&eb)[5],
                                              T (&gc)[NCORE], T (&gam)[9]) {
    const T p1 = eb[0] - g[LE + 0], p6 = g[LE + 1] - eb[1], p5 = g[LE + 2] - eb[2], p3 = eb[3] - g[LE + 3],
            p7 = eb[4] - g[LE + 4], pv = ea4 - g[LE + 4];
    T gl = g[LL];
    gl = cond_fma(f(CF_L1), p1, gl);
    gl = cond_fma(f(CF_L3), p3, gl);
    gl = cond_fma(f(CF_L5), p5, gl);
    gl = cond_fma(f(CF_L6), p6, gl);
    gl = cond_fma(f(CF_L7), p7, gl);
    gc[4] = gl;
    gc[5] = cond_fma(f(CF_VV), pv, cond_fma(-f(CF_HV), g[LS], g[LV]));
    gc[0] = g[0];
    gc[1] = cond_fma(f(CF_MC + 0), p1, g[1]);
    gc[2] = cond_fma(f(CF_MC + 2), p3, g[3]);
    gc[3] = cond_fma(-f(CF_HT), g[LS], g[LT]);
    gam[0] = g[2];
    gam[1] = g[4];
    gam[2] = cond_fma(f(CF_MC + 4), p5, g[5]);
    gam[3] = cond_fma(f(CF_MC + 5), p6, g[6]);
    gam[4] = cond_fma(f(CF_MC + 6), p7, g[7]);
    gam[5] = g[8];
    gam[6] = g[LY + 1];
    gam[7] = cond_fma(f(CF_W0), pv, g[LY]);
    gam[8] = g[LY + 2];
    gc[6] = cond_fma(f(CF_Y23), gam[8], g[LY + 3]);
    gc[0] = cond_fma(f(CF_X + 0), gam[0], gc[0]);
    gc[1] = cond_fma(f(CF_X + 1), gam[0], gc[1]);
    gc[3] = cond_fma(f(CF_X + 2), gam[0], gc[3]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        T a = gc[q];
#pragma unroll
        for (int k = 0; k < 5; ++k) a = cond_fma(f(CF_X + 3 + 4 * k + q), gam[1 + k], a);
        a = cond_fma(f(CF_Y1 + q), gam[6], a);
        a = cond_fma(f(CF_Y0 + q), gam[7], a);
        gc[q] = cond_fma(f(CF_Y2 + q), gam[8], a);
    }
}

// J^T: from the core multipliers w (rows a, b, c, d, N, O, E), every row's: the transpose of
// cond_reduce.  dl: the stage's multipliers of rows b, c, d, E less those of the stage below;
// dg: its multipliers of the vapour links (CO2, H2O, N2, enthalpy) less those of the stage above.
template <class T>
__device__ inline void cond_expand_t(const CondRef<const T>& f, const T (&g)[NV], const T (&w)[NCORE],
                                              const T (&dl)[4], const T (&dg)[4], const T (&gam)[9], T (&v)[NR]) {
    v[0] = w[0];
    v[1] = g[LE + 0] + (w[0] + w[1]);
    v[2] = w[1];
    v[3] = g[LE + 3] + ((w[0] + w[2]) - w[3]);
    v[4] = w[2];
    v[5] = (w[3] - w[1]) - g[LE + 2];
    v[6] = (w[2] - w[1]) - g[LE + 1];
    v[7] = g[LE + 4] + ((w[1] + w[2]) - w[3]);
    v[8] = w[3];
    v[9] = w[4];
    v[10] = w[5];
    v[R_E] = w[6];
    v[R_H] = g[LS];
    T p2 = cond_fma(-f(CF_MC + 1), dl[0], cond_fma(-f(CF_H2), dl[3], gam[0]));
    T p4 = cond_fma(-f(CF_MC + 3), dl[1], cond_fma(-f(CF_H4), dl[3], gam[1]));
    T p5 = cond_fma(-f(CF_MC + 4), dl[2] - dl[0], cond_fma(-f(CF_H5), dl[3], gam[2]));
    T p6 = cond_fma(-f(CF_MC + 5), dl[1] - dl[0], cond_fma(-f(CF_H6), dl[3], gam[3]));
    T p7 = cond_fma(-f(CF_MC + 6), (dl[0] + dl[1]) - dl[2], cond_fma(-f(CF_H7), dl[3], gam[4]));
    T p8 = cond_fma(-f(CF_MC + 7), dl[2], cond_fma(-f(CF_H8), dl[3], gam[5]));
    T y1 = cond_fma(-f(CF_W1), dg[1], cond_fma(-f(CF_Z0 + 1), dg[3], gam[6]));
    T y0 = cond_fma(-f(CF_W0), dg[0], cond_fma(-f(CF_Z0 + 0), dg[3], gam[7]));
    const T y2 = cond_fma(-f(CF_W2), dg[2], cond_fma(-f(CF_Z0 + 2), dg[3], gam[8]));
    v[R_SY] = f(CF_IY2) * y2;
    y0 = cond_fma(-f(CF_D0), y2, y0);
    y1 = cond_fma(-f(CF_D1), y2, y1);
    v[R_VC] = f(CF_IY0) * y0;
    p4 = cond_fma(-f(CF_K4 + 0), y0, p4);
    p5 = cond_fma(-f(CF_K4 + 1), y0, p5);
    p6 = cond_fma(-f(CF_K4 + 2), y0, p6);
    p7 = cond_fma(-f(CF_K4 + 3), y0, p7);
    p8 = cond_fma(-f(CF_K4 + 4), y0, p8);
    v[R_VH] = f(CF_IY1) * y1;
    p8 = cond_fma(-f(CF_H18), y1, p8);
    p8 = cond_fma(f(CF_X48), p4, p8);
    p8 = cond_fma(f(CF_X58), p5, p8);
    p8 = cond_fma(f(CF_X68), p6, p8);
    p8 = cond_fma(f(CF_X78), p7, p8);
    v[R_SX] = f(CF_I8) * p8;
    p2 = cond_fma(-f(CF_C2), p8, p2);
    p4 = cond_fma(-f(CF_C4), p8, p4);
    p5 = cond_fma(-f(CF_C5), p8, p5);
    p6 = cond_fma(-f(CF_C6), p8, p6);
    p7 = cond_fma(-f(CF_C7), p8, p7);
    v[R_RX + 4] = f(CF_I57) * p7;
    p2 = cond_fma(-f(CF_A52), p7, p2);
    p4 = cond_fma(-f(CF_A54), p7, p4);
    v[R_RX + 1] = f(CF_I26) * p6;
    p4 = cond_fma(-f(CF_A24), p6, p4);
    p2 = cond_fma(-f(CF_A22), p6, p2);
    v[R_RX + 2] = f(CF_I35) * p5;
    p2 = cond_fma(-f(CF_A32), p5, p2);
    v[R_RX + 3] = f(CF_I44) * p4;
    v[R_RX] = f(CF_I12) * p2;
}

// ---- factorization -------------------------------------------------------------------------

// own Jacobian entries of a stage, in T
template <class T>
struct OwnEntries {
    const double* j;   // the stage's segment at the scenario
    int64_t ld;
    int t;
    __device__ __forceinline__ T operator()(int r, int lv) const { return (T)j[(int64_t)c_slotJ[t][r][lv] * ld]; }
};

// a = b to 2^12 units in the last place (4.5e-13 to 9e-13 relative: values computed in another order
// of the same operations agree to a few), or both zero; on the integer pipe
__device__ __forceinline__ bool alike(double a, double b) {
    const unsigned long long x = (unsigned long long)__double_as_longlong(a),
                             y = (unsigned long long)__double_as_longlong(b);
    return x - y + 4096ull <= 8192ull || ((x | y) << 1) == 0ull;
}
__device__ __forceinline__ bool opposite(double a, double b) { return alike(a, -b); }
// Whether the values that the condensation of a stage assumes instead of reading are there.  Every load
// is issued at once: no condition skips one.
__device__ __forceinline__ bool condense_conforms(const double* __restrict__ jac, int64_t ld, int s, int n) {
    const int t = stage_type(n);
    const OwnEntries<double> A{jac + (int64_t)c_segJ[n] * ld + s, ld, t};
    int ok = alike(A(R_H, LS), 1.0);
    static_for<0, 9>([&](auto C) {
        constexpr int c = decltype(C)::value;
        static_for<0, 5>([&](auto K) {
            constexpr int k = decltype(K)::value;
            if constexpr (nu(c, k) != 0)
                ok &= alike(A(c, LE + k), -nu(c, k));
        });
    });
    const int below = n > 0 ? n - 1 : 0, above = n + 1 < N_STAGES ? n + 1 : N_STAGES - 1;
    const OwnEntries<double> B{jac + (int64_t)c_segJ[below] * ld + s, ld, stage_type(below)},
        U{jac + (int64_t)c_segJ[above] * ld + s, ld, stage_type(above)};
    if (n > 0) {   // its liquid in the rows of the stage below
        static_for<0, 9>([&](auto C) {
            constexpr int c = decltype(C)::value;
            ok &= opposite(A(c, c), B(c, AX + c));
            ok &= opposite(A(c, LL), B(c, AL));
            ok &= opposite(A(R_E, c), B(R_E, AX + c));
        });
        ok &= opposite(A(R_E, LL), B(R_E, AL));
    }
    if (n + 1 < N_STAGES) {   // its vapour in the rows of the stage above
        static_for<0, 4>([&](auto J) {
            constexpr int j = decltype(J)::value;
            ok &= opposite(A(7 + j, LY + j), U(7 + j, BY + j));
            ok &= opposite(A(7 + j, LV), U(7 + j, BV));
            ok &= opposite(A(R_E, LY + j), U(R_E, BY + j));
        });
        ok &= opposite(A(R_E, LV), U(R_E, BV));
        if (n > 0) {   // the shares of its energy row's dT in the neighbours' rows, and their sum
            const double a = A(R_E, LT), l = B(R_E, AT), v = U(R_E, BT);
            ok &= fabs(a + v + l) <= 0x1p-40 * (fabs(v) + fabs(l));
        }
    }
    return ok;
}

// Every (scenario, stage) condensed, one thread each: about 330 multiply-adds, all stages at
// once.  mask (optional): only scenarios with mask[s] != 0.  skip (optional, device): the
// stored values are those of this Jacobian.  CHECK (a Jacobian from outside the library): *odd is set
// where the condensation does not hold, by blocks of their own next to those that condense the same
// stage (its entries come from L2; on the same threads their loads cost up to twice as much): kkt_factor
// of 20000 scenarios FP64 700 -> 727 us, FP32 157 -> 173, of up to 500 the same.  Grid (ceil(S / 64),
// N_STAGES, with CHECK twice that), 64 threads.
template <class T, bool CHECK>
__global__ void __launch_bounds__(64) condense_kernel(int S, int64_t ld, const BView b, const double* __restrict__ jac,
                                                      T* __restrict__ F, const int* __restrict__ mask,
                                                      const int* __restrict__ skip, int* __restrict__ odd) {
    if (skip && *skip) return;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = CHECK ? blockIdx.y >> 1 : blockIdx.y;
    if (live_prob(b, s, S, PS_ACT) < 0 || (mask && mask[s] == 0)) return;
    if (CHECK && (blockIdx.y & 1)) {
        if (!condense_conforms(jac, ld, s, n)) *odd = 1;
        return;
    }
    const int t = stage_type(n);
    const OwnEntries<T> A{jac + (int64_t)c_segJ[n] * ld + s, ld, t};
    // the energy row's dT: the liquid's share from the stage below's row, the vapour's from the
    // stage above's
    const T tot = A(R_E, LT);
    T Lt, Vt;
    if (n > 0) {
        Lt = -(T)jac[(int64_t)(c_segJ[n - 1] + c_slotJ[stage_type(n - 1)][R_E][AT]) * ld + s];
        Vt = tot - Lt;
    } else {
        Vt = -(T)jac[(int64_t)(c_segJ[1] + c_slotJ[1][R_E][BT]) * ld + s];
        Lt = tot - Vt;
    }
    const bool safe = condense_stage<T>(A, Lt, Vt, cond_ref(F, ld, n, s));
    if (CHECK && !safe) *odd = 1;
}

// the magnitude order of a pivot candidate: for FP64 by the high word (a relative 2^-20)
__device__ __forceinline__ unsigned core_key(double a) { return (unsigned)__double2hiint(a) & 0x7fffffffu; }
__device__ __forceinline__ unsigned core_key(float a) { return __float_as_uint(a) & 0x7fffffffu; }
__device__ __forceinline__ double core_mag(unsigned k, double) { return __hiloint2double((int)k, 0); }
__device__ __forceinline__ float core_mag(unsigned k, float) { return __uint_as_float(k); }

// |a| > tiny >= 0, false for NaN; FP64 on the integer pipe (the order of the bits)
__device__ __forceinline__ bool core_above(double a, double tiny) {
    const long long m = __double_as_longlong(a) & 0x7fffffffffffffffll;
    return m > __double_as_longlong(tiny) && m <= (0x7ffll << 52);
}
__device__ __forceinline__ bool core_above(float a, float tiny) { return fabsf(a) > tiny; }

__host__ __device__ constexpr size_t chain_smem(size_t es, int spb, int cg) {
    // N At^-1 (7 x 5), two pivot-column buffers (7 + reciprocal), pivot rows, column maxima
    return (size_t)spb * (51 * es + (2 + 2 * cg) * sizeof(int));
}

// The chain over the stages: At_n from the stored M, N and the stage below's K, its inverse by
// in-place Gauss-Jordan with partial pivoting, then K, D, T.  SPB scenarios per block, CG
// threads per scenario, thread (scenario i, group g) at threadIdx.x = g SPB + i holding the
// core's columns g, g + CG, ... in registers; a step's pivot column travels through shared
// memory (one barrier per step, two buffers).  The chain is ten dependent inverses of seven
// dependent steps: latency bounds it, FP64's (64 cycles per multiply-add and warp) most of all, so a
// scenario's columns are spread over lanes and small blocks over all SMs.  FP64 82 us up to 500 scenarios
// (a warp's block LU of 22 x 22 blocks: 400), 560 at 20000 (8900); FP32 28 us at 5000 (252).
template <class T, int SPB, int CG>
__global__ void __launch_bounds__(SPB * CG) chain_kernel(int S, int64_t ld, const BView b, T* F, int* __restrict__ sing,
                                                         double pivtol, const int* __restrict__ mask,
                                                         const int* __restrict__ skip) {
    if (skip && *skip) return;
    constexpr int NCOL = (NCORE + CG - 1) / CG;
    extern __shared__ __align__(16) unsigned char chain_sm[];
    T* sN = reinterpret_cast<T*>(chain_sm);             // [7][5][SPB]
    T* sP = sN + 35 * SPB;                              // [2][8][SPB]
    int* sR = reinterpret_cast<int*>(sP + 2 * 8 * SPB); // [2][SPB] pivot rows
    unsigned* sK = reinterpret_cast<unsigned*>(sR + 2 * SPB);   // [2][CG][SPB] column maxima
    const int i = (int)threadIdx.x % SPB, g = (int)threadIdx.x / SPB;
    const int s = blockIdx.x * SPB + i;
    const bool live = live_prob(b, s, S, PS_ACT) >= 0 && !(mask && mask[s] == 0);
    if (!__syncthreads_or(live)) return;
    int bad = 0;
    T kc[5][5];   // K of the stage below
    // the thread's columns of a stage's M and N: loaded a stage ahead, so that the elimination
    // does not start with a wait for memory
    T cm[NCOL][5], ce[NCOL][5];
    auto columns = [&](int n) {
        const CondRef<T> f = cond_ref(F, ld, n, (int64_t)s);
#pragma unroll
        for (int c = 0; c < NCOL; ++c) {
            const int j = g + CG * c;
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                cm[c][k] = j < 5 ? f(CF_M + 5 * k + (j < 5 ? j : 0)) : T(0);
                ce[c][k] = (j < NCORE && j != 4) ? f(CF_N + 6 * k + (j < 4 ? j : (j < NCORE ? j - 1 : 0))) : T(0);
            }
        }
    };
    columns(0);
#pragma unroll 1
    for (int n = 0; n < N_STAGES; ++n) {
        const CondRef<T> f = cond_ref(F, ld, n, (int64_t)s);
        T M[5][5], N[5][6];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
#pragma unroll
            for (int j = 0; j < 5; ++j) M[k][j] = m_has(k, j) ? f(CF_M + 5 * k + j) : T(0);
#pragma unroll
            for (int j = 0; j < 6; ++j) N[k][j] = n_has(k, j) ? f(CF_N + 6 * k + j) : T(0);
        }
        if (n > 0) {
#pragma unroll
            for (int k = 0; k < 5; ++k)
#pragma unroll
                for (int q = 0; q < 5; ++q) kc[q][k] = sN[(e_row(k) * 5 + q) * SPB + i];
        }
        T a[NCOL][NCORE];
        unsigned km = 0u;
#pragma unroll
        for (int c = 0; c < NCOL; ++c) {
            const int j = g + CG * c;
            T m[5], e[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                m[k] = cm[c][k];
                e[k] = ce[c][k];
            }
            if (n > 0) {
#pragma unroll
                for (int q = 0; q < 5; ++q)
#pragma unroll
                    for (int k = 0; k < 5; ++k) e[q] = cond_fma(-kc[q][k], m[k], e[q]);
            }
            a[c][0] = m[0];
            a[c][1] = m[1] + e[0];
            a[c][2] = m[2] + e[0];
            a[c][3] = m[3] + (e[1] - e[0]);
            a[c][4] = e[2];
            a[c][5] = e[3];
            a[c][6] = m[4] + e[4];
            if (j < NCORE)
#pragma unroll
                for (int r = 0; r < NCORE; ++r) km = max(km, core_key(a[c][r]));
        }
        sK[((n & 1) * CG + g) * SPB + i] = km;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < CG; ++q) km = max(km, sK[((n & 1) * CG + q) * SPB + i]);
        if (n + 1 < N_STAGES) columns(n + 1);
        const T tiny = (T)pivtol * core_mag(km, T(0));
        unsigned orig = 0x6543210u;   // nibble k: the row now at position k
#pragma unroll
        for (int k = 0; k < NCORE; ++k) {
            T fc[NCORE], piv = T(0);
            int p = k;
            const bool own = g == k % CG;
            if (own) {
                T(&c)[NCORE] = a[k / CG];
                unsigned best = core_key(c[k]);
#pragma unroll
                for (int r = k + 1; r < NCORE; ++r) {
                    const unsigned v = core_key(c[r]);
                    p = v > best ? r : p;
                    best = max(v, best);
                }
                T pv = c[k];
#pragma unroll
                for (int r = k + 1; r < NCORE; ++r) {
                    const T x = c[r];
                    c[r] = p == r ? pv : x;
                    pv = p == r ? x : pv;
                }
                if (!core_above(pv, tiny)) {   // too small, or NaN
                    bad = 1;
                    pv = (pv < T(0) ? T(-1) : T(1)) * (tiny > T(0) ? tiny : T(1));
                }
                piv = cond_recip(pv);
                c[k] = pv;
#pragma unroll
                for (int r = 0; r < NCORE; ++r) fc[r] = c[r];
            }
            T* bp = sP + (k & 1) * 8 * SPB;
            if (own) {
#pragma unroll
                for (int r = 0; r < NCORE; ++r)
                    if (r != k) bp[r * SPB + i] = fc[r];
                bp[7 * SPB + i] = piv;
                sR[(k & 1) * SPB + i] = p;
            }
            __syncthreads();
            if (!own) {
#pragma unroll
                for (int r = 0; r < NCORE; ++r) fc[r] = r != k ? bp[r * SPB + i] : T(0);
                piv = bp[7 * SPB + i];
                p = sR[(k & 1) * SPB + i];
            }
            // rows k and p change places, row k scales by the pivot's reciprocal, the others subtract
            // their multiple of it; the pivot column itself starts from the unit vector (one code
            // path for all columns: no divergence inside a warp)
#pragma unroll
            for (int c = 0; c < NCOL; ++c) {
                const bool unit = own && c == k / CG;
                T u = a[c][k];
#pragma unroll
                for (int r = k + 1; r < NCORE; ++r) {
                    const T x = a[c][r];
                    const bool h = p == r && !unit;
                    a[c][r] = h ? u : x;
                    u = h ? x : u;
                }
                u = (unit ? T(1) : u) * piv;
#pragma unroll
                for (int r = 0; r < NCORE; ++r)
                    if (r != k) a[c][r] = cond_fma(-fc[r], u, unit ? T(0) : a[c][r]);
                a[c][k] = u;
            }
            const unsigned x = ((orig >> (4 * k)) ^ (orig >> (4 * p))) & 15u;
            orig ^= (x << (4 * k)) | (x << (4 * p));
        }
        // the column at position j is the inverse's column of row orig[j]
#pragma unroll
        for (int c = 0; c < NCOL; ++c) {
            const int j = g + CG * c;
            if (j >= NCORE) continue;
            const int r = (int)((orig >> (4 * j)) & 15u);
            if (live)
#pragma unroll
                for (int q = 0; q < NCORE; ++q) f(CF_INV + NCORE * q + r) = a[c][q];
            T w[5];
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                T v = T(0);
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    if (n_has(q, k)) v = cond_fma(N[q][k], a[c][n_core(k)], v);
                w[q] = v;
            }
#pragma unroll
            for (int q = 0; q < 5; ++q) sN[(r * 5 + q) * SPB + i] = w[q];
            if (live) {
                if (r >= 3)
#pragma unroll
                    for (int q = 0; q < 5; ++q) f(CF_D + 5 * q + r - 2) = w[q];
                if (r < 4 || r == 6) {
                    const int k = r < 4 ? r : 4;
#pragma unroll
                    for (int q = 0; q < 5; ++q) {
                        T v = T(0);
#pragma unroll
                        for (int z = 0; z < 5; ++z)
                            if (m_has(q, z)) v = cond_fma(M[q][z], a[c][z], v);
                        f(CF_T + 5 * q + k) = v;
                    }
                }
            }
        }
        __syncthreads();
        if (g == CG - 1 && live)
#pragma unroll
            for (int q = 0; q < 5; ++q)
                f(CF_D + 5 * q) = (sN[(5 + q) * SPB + i] + sN[(10 + q) * SPB + i]) - sN[(15 + q) * SPB + i];
    }
    __syncthreads();
    sK[g * SPB + i] = (unsigned)bad;
    __syncthreads();
    for (int q = 0; q < CG; ++q) bad |= (int)sK[q * SPB + i];
    if (live && g == 0 && sing) sing[s] = bad;
}

// ---- block solves ----------------------------------------------------------------------------
// The solve kernels: 6 scenarios x 10 stages on the 60 first threads of a two-warp block (scenario
// fastest, so an access covers 48 consecutive bytes of an entry in FP64).  Neighbouring stages
// exchange through shared memory; the chains run on the 30 first lanes of the first warp, a lane
// per scenario and link quantity.  Small blocks because FP64 instructions bound these kernels and
// 5000 scenarios are few: 834 blocks share out evenly over 152 SMs (32 scenarios x 10 stages per
// block left five SMs with twice the others' work), and ten scenarios already use two SMs.  More per
// block coalesce better, but their chains take longer: a solve, direction and residual of 35000 scenarios
// with 6 / 8 / 16 / 32 take 784 / 791 / 781 / 920 us in FP32, 1070 / 1185 / 1336 / 1566 in FP64; of 5000
// 182 / 210 / 209 / 243 in FP32.  Six blocks of 168 registers per SM (eight of 128: 843 us at 35000).
constexpr int CS_N = 6;
constexpr int CS_T = 64;
constexpr int CS_LINK = NLINK * NLINK * CS_N;    // link map of a stage
constexpr int CS_VEC = NLINK * CS_N;             // link quantities of a stage
constexpr int CS_EX = 8 * CS_N;                  // exchanged values of a stage
static_assert(CS_N * N_STAGES <= CS_T && CS_N * NLINK <= 32, "the block's threads and its chain lanes");

// the thread's place: stage n, scenario slot i of the block, scenario s; the threads past the 60th
// repeat places of the last stage (same values to the same shared memory, no global stores)
struct CondPlace {
    int n, i, s, pr;
    int64_t o;       // a scenario of the problem arrays (s, or the last one past the end)
    bool live;
    __device__ __forceinline__ CondPlace(int S, const BView& b) {
        const int t = threadIdx.x;
        const bool slot = t < CS_N * N_STAGES;
        n = slot ? t / CS_N : N_STAGES - 1;
        i = slot ? t - n * CS_N : t - CS_N * N_STAGES;
        s = blockIdx.x * CS_N + i;
        pr = live_prob(b, s, S, PS_ACT);
        live = slot && pr >= 0;
        o = s < S ? s : S - 1;
    }
};
__host__ __device__ constexpr size_t cond_smem(size_t es) {
    return es * (size_t)N_STAGES * (CS_LINK + 2 * CS_VEC + CS_EX);
}

// v_n += D_n v_prev along the column (UP: prev = n - 1, n = 1..8; else prev = n + 1, n = 8..1), the
// maps d transposed with TR; the block's first warp, a lane per scenario and quantity.  The maps are
// in registers before the first step.
template <class T, bool TR, bool UP>
__device__ __forceinline__ void link_chain(const T* d, T* v) {
    if (threadIdx.x >= 32) return;
    const int q = (int)threadIdx.x / CS_N, i = (int)threadIdx.x - q * CS_N;   // q = 5: idle
    const int qq = q < NLINK ? q : 0;
    T m[8][NLINK];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int n = UP ? k + 1 : 8 - k;
#pragma unroll
        for (int j = 0; j < NLINK; ++j) m[k][j] = d[n * CS_LINK + (TR ? j * NLINK + qq : qq * NLINK + j) * CS_N + i];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int n = UP ? k + 1 : 8 - k;
        const T* w = v + (UP ? n - 1 : n + 1) * CS_VEC + i;
        T a = v[n * CS_VEC + qq * CS_N + i], c;
        a = cond_fma(m[k][0], w[0], a);
        c = m[k][1] * w[CS_N];
        a = cond_fma(m[k][2], w[2 * CS_N], a);
        c = cond_fma(m[k][3], w[3 * CS_N], c);
        a = cond_fma(m[k][4], w[4 * CS_N], a);
        if (q < NLINK) v[n * CS_VEC + q * CS_N + i] = a + c;
        __syncwarp();
    }
}

template <class T>
__device__ __forceinline__ void stage_links(const CondRef<const T>& f, int field, T* d, int n, int lane) {
#pragma unroll
    for (int e = 0; e < NLINK * NLINK; ++e) d[n * CS_LINK + e * CS_N + lane] = f(field + e);
}

// u = J^-1 r at the thread's (scenario, stage): every thread of the block takes part (its own
// values are meaningless where the scenario's factors are not)
template <class T>
__device__ __forceinline__ void cond_solve_block(const T* __restrict__ F, int64_t ld, int64_t s, int n, int lane,
                                                 const T (&r)[NR], T* sm, T (&u)[NV]) {
    T* sd = sm;
    T* sg = sd + N_STAGES * CS_LINK;
    T* sl = sg + N_STAGES * CS_VEC;
    T* sx = sl + N_STAGES * CS_VEC;
    const CondRef<const T> f = cond_ref(F, ld, n, s);
    stage_links(f, CF_D, sd, n, lane);
    T rc[NCORE], rho[9], lo[4], go[4];
    cond_reduce(f, r, rc, rho, lo, go);
    T* x = sx + n * CS_EX + lane;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        x[CS_N * k] = lo[k];
        x[CS_N * (4 + k)] = go[k];
    }
    __syncthreads();
    if (n + 1 < N_STAGES) {
        const T* xa = x + CS_EX;
        rc[1] += xa[0];
        rc[2] += xa[CS_N];
        rc[3] += xa[2 * CS_N];
        rc[6] += xa[3 * CS_N];
    }
    if (n > 0) {
        const T* xb = x - CS_EX;
        rc[1] += xb[4 * CS_N];
        rc[2] += xb[4 * CS_N];
        rc[3] += xb[5 * CS_N] - xb[4 * CS_N];
        rc[4] += xb[6 * CS_N];
        rc[6] += xb[7 * CS_N];
    }
    T t[NCORE];
    auto core = [&]() {
#pragma unroll
        for (int c = 0; c < NCORE; ++c) {
            T a = f(CF_INV + NCORE * c) * rc[0];
#pragma unroll
            for (int q = 1; q < NCORE; ++q) a = cond_fma(f(CF_INV + NCORE * c + q), rc[q], a);
            t[c] = a;
        }
    };
    core();
#pragma unroll
    for (int q = 0; q < NLINK; ++q) {
        T a = T(0);
#pragma unroll
        for (int k = 0; k < 6; ++k)
            if (n_has(q, k)) a = cond_fma(f(CF_N + 6 * q + k), t[n_core(k)], a);
        sg[n * CS_VEC + q * CS_N + lane] = a;
    }
    __syncthreads();
    link_chain<T, false, true>(sd, sg);
    __syncthreads();
    stage_links(f, CF_T, sd, n, lane);
    if (n > 0) {
        const T* g = sg + (n - 1) * CS_VEC + lane;
        rc[1] += g[0];
        rc[2] += g[0];
        rc[3] += g[CS_N] - g[0];
        rc[4] += g[2 * CS_N];
        rc[5] += g[3 * CS_N];
        rc[6] += g[4 * CS_N];
        core();
    }
#pragma unroll
    for (int q = 0; q < NLINK; ++q) {
        T a = T(0);
#pragma unroll
        for (int k = 0; k < 5; ++k)
            if (m_has(q, k)) a = cond_fma(f(CF_M + 5 * q + k), t[k], a);
        sl[n * CS_VEC + q * CS_N + lane] = a;
    }
    __syncthreads();
    link_chain<T, false, false>(sd, sl);
    __syncthreads();
    if (n + 1 < N_STAGES) {
        const T* l = sl + (n + 1) * CS_VEC + lane;
#pragma unroll
        for (int k = 0; k < NLINK; ++k) {
            const T lk = l[CS_N * k];
#pragma unroll
            for (int c = 0; c < NCORE; ++c) t[c] = cond_fma(f(CF_INV + NCORE * c + e_row(k)), lk, t[c]);
        }
    }
    T fl[6], fa[5], vb = T(0);
    cond_expand(f, t, rho, u, fl);
#pragma unroll
    for (int k = 0; k < 6; ++k) x[CS_N * k] = fl[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 5; ++k) fa[k] = n + 1 < N_STAGES ? x[CS_EX + CS_N * k] : T(0);
    if (n > 0) vb = x[5 * CS_N - CS_EX];
    cond_extents(f, r, fl, fa, vb, u);
}

// v = J^-T g likewise
template <class T>
__device__ __forceinline__ void cond_solve_t_block(const T* __restrict__ F, int64_t ld, int64_t s, int n, int lane,
                                                   const T (&g)[NV], T* sm, T (&v)[NR]) {
    T* sd = sm;
    T* sg = sd + N_STAGES * CS_LINK;
    T* sl = sg + N_STAGES * CS_VEC;
    T* sx = sl + N_STAGES * CS_VEC;
    const CondRef<const T> f = cond_ref(F, ld, n, s);
    stage_links(f, CF_T, sd, n, lane);
    T* x = sx + n * CS_EX + lane;
#pragma unroll
    for (int k = 0; k < 5; ++k) x[CS_N * k] = g[LE + k];
    __syncthreads();
    T eb[5], gc[NCORE], gam[9];
#pragma unroll
    for (int k = 0; k < 5; ++k) eb[k] = n > 0 ? x[CS_N * k - CS_EX] : T(0);
    cond_reduce_t(f, g, n + 1 < N_STAGES ? x[4 * CS_N + CS_EX] : T(0), eb, gc, gam);
#pragma unroll
    for (int k = 0; k < NLINK; ++k) {
        T a = f(CF_INV + e_row(k)) * gc[0];
#pragma unroll
        for (int c = 1; c < NCORE; ++c) a = cond_fma(f(CF_INV + NCORE * c + e_row(k)), gc[c], a);
        sg[n * CS_VEC + k * CS_N + lane] = a;
    }
    __syncthreads();
    link_chain<T, true, true>(sd, sg);
    __syncthreads();
    stage_links(f, CF_D, sd, n, lane);
    if (n > 0) {
        const T* a = sg + (n - 1) * CS_VEC + lane;
#pragma unroll
        for (int q = 0; q < NLINK; ++q) {
            const T aq = a[CS_N * q];
#pragma unroll
            for (int k = 0; k < 5; ++k)
                if (m_has(q, k)) gc[k] = cond_fma(f(CF_M + 5 * q + k), aq, gc[k]);
        }
    }
    T w[NCORE];
    auto core = [&]() {
#pragma unroll
        for (int q = 0; q < NCORE; ++q) {
            T a = f(CF_INV + q) * gc[0];
#pragma unroll
            for (int c = 1; c < NCORE; ++c) a = cond_fma(f(CF_INV + NCORE * c + q), gc[c], a);
            w[q] = a;
        }
    };
    core();
    T* bl = sl + n * CS_VEC + lane;
    bl[0] = (w[1] + w[2]) - w[3];
    bl[CS_N] = w[3];
    bl[2 * CS_N] = w[4];
    bl[3 * CS_N] = w[5];
    bl[4 * CS_N] = w[6];
    __syncthreads();
    link_chain<T, true, false>(sd, sl);
    __syncthreads();
    T ba[4] = {T(0), T(0), T(0), T(0)};
    if (n + 1 < N_STAGES) {
        const T* bn = bl + CS_VEC;
#pragma unroll
        for (int q = 0; q < NLINK; ++q) {
            const T bq = bn[CS_N * q];
            if (q != 3) ba[q < 3 ? q : 3] = bq;
#pragma unroll
            for (int k = 0; k < 6; ++k)
                if (n_has(q, k)) gc[n_core(k)] = cond_fma(f(CF_N + 6 * q + k), bq, gc[n_core(k)]);
        }
        core();
    }
    x[0] = w[1];
    x[CS_N] = w[2];
    x[2 * CS_N] = w[3];
    x[3 * CS_N] = w[6];
    __syncthreads();
    T dl[4] = {w[1], w[2], w[3], w[6]};
    if (n > 0)
#pragma unroll
        for (int k = 0; k < 4; ++k) dl[k] -= x[CS_N * k - CS_EX];
    const T dg[4] = {((w[1] + w[2]) - w[3]) - ba[0], w[3] - ba[1], w[4] - ba[2], w[6] - ba[3]};
    cond_expand_t(f, g, w, dl, dg, gam, v);
}

// the design column: q = J^-1 b, b = dc/dtheta nonzero in the hydraulic rows only, whose slack
// (coefficient 1) nothing else contains: q is -u_max pi theta / 2 at the slacks of the section's
// stages and zero elsewhere
__device__ __forceinline__ double slack_q(const Params& P, const double* x, int64_t ld, int sec, int NP, int pr) {
    return -P.u_max * M_PI * 0.5 * x[(int64_t)NSC * ld + (int64_t)sec * NP + pr];
}

// Schur sums of a factorization (H = W + Sigma, W has no slack entries): planes [0] q^T H q, [1]
// q^T q, [4] the d-d Hessian entry of the first section, [6], [7], [8] those of the second (two
// sections), [5] the singular flag, [2], [3] the given right-hand side's sums (or 0)
__device__ __forceinline__ void store_schur(const Params& P, const double* __restrict__ sig,
                                            const double* __restrict__ hes, bool use_w, const int* __restrict__ sing,
                                            double qs, double r2, double r3, double* part, int64_t ld, int64_t s, int n) {
    const double a = qs * (sig[(int64_t)(NV * n + LS) * ld + s] * qs), q2 = qs * qs;
    const bool top = stage_sec(n, P.nsec) == 1;
    double w[9] = {top ? 0.0 : a, top ? 0.0 : q2, r2, r3, 0.0, 0.0, top ? a : 0.0, top ? q2 : 0.0, 0.0};
    if (n == 0) {
        if (use_w) {
            w[4] = hes[(int64_t)(NHS * N_STAGES) * ld + s];
            if (P.nsec == 2) w[8] = hes[(int64_t)(NHS * N_STAGES + 1) * ld + s];
        }
        if (sing) w[5] = (double)sing[s];
    }
    if (P.nsec == 2) store_partials<9>(w, part, ld, (int)s, n);
    else {
        const double w6[6] = {w[0], w[1], w[2], w[3], w[4], w[5]};
        store_partials<6>(w6, part, ld, (int)s, n);
    }
}

__global__ void __launch_bounds__(128) cond_schur_kernel(const Params P, int S, int64_t ld, const BView b,
                                                         const double* __restrict__ x, const double* __restrict__ sig,
                                                         const double* __restrict__ hes, bool use_w,
                                                         const int* __restrict__ sing, double* part) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = blockIdx.y;
    const int pr = live_prob(b, s, S, PS_ACT);
    if (pr < 0) return;
    store_schur(P, sig, hes, use_w, sing, slack_q(P, x, ld, stage_sec(n, P.nsec), b.NP, pr), 0.0, 0.0, part, ld, s, n);
}

// factors of the solve kernels: FP32, FP64, or mixed (esc[s] != 0: the scenario's are FP64)
struct CondFac {
    const float* f32;
    const double* f64;
    const int* esc;
};
enum { CP_FP64 = 0, CP_FP32 = 1, CP_MIXED = 2 };

// o = J^-1 r (r, o doubles) in the factors' precision
template <int PREC>
__device__ __forceinline__ void cond_solve_prec(const CondFac& K, int64_t ld, const CondPlace& at,
                                                const double (&r)[NR], unsigned char* sm, double (&o)[NV]) {
    if constexpr (PREC != CP_FP64) {
        float rf[NR], uf[NV];
#pragma unroll
        for (int j = 0; j < NR; ++j) rf[j] = (float)r[j];
        cond_solve_block<float>(K.f32, ld, at.o, at.n, at.i, rf, (float*)sm, uf);
#pragma unroll
        for (int j = 0; j < NV; ++j) o[j] = (double)uf[j];
    }
    if constexpr (PREC != CP_FP32) {
        const bool mine = PREC == CP_FP64 || (at.live && K.esc[at.s] != 0);
        if (PREC == CP_FP64 || __syncthreads_or(mine)) {
            double u[NV];
            cond_solve_block<double>(K.f64, ld, at.o, at.n, at.i, r, (double*)sm, u);
            if (mine)
#pragma unroll
                for (int j = 0; j < NV; ++j) o[j] = u[j];
        }
    }
}
template <int PREC>
__device__ __forceinline__ void cond_solve_t_prec(const CondFac& K, int64_t ld, const CondPlace& at,
                                                  const double (&g)[NV], unsigned char* sm, double (&o)[NR]) {
    if constexpr (PREC != CP_FP64) {
        float gf[NV], vf[NR];
#pragma unroll
        for (int j = 0; j < NV; ++j) gf[j] = (float)g[j];
        cond_solve_t_block<float>(K.f32, ld, at.o, at.n, at.i, gf, (float*)sm, vf);
#pragma unroll
        for (int j = 0; j < NR; ++j) o[j] = (double)vf[j];
    }
    if constexpr (PREC != CP_FP32) {
        const bool mine = PREC == CP_FP64 || (at.live && K.esc[at.s] != 0);
        if (PREC == CP_FP64 || __syncthreads_or(mine)) {
            double v[NR];
            cond_solve_t_block<double>(K.f64, ld, at.o, at.n, at.i, g, (double*)sm, v);
            if (mine)
#pragma unroll
                for (int j = 0; j < NR; ++j) o[j] = v[j];
        }
    }
}

// p = J^-1 r_c, and with planes the Schur sums of the right-hand side (r_z, r_c): 1 -- planes [2]
// q^T (r_z - H p), [3] q^T p of the first section, [0], [1] of the second; 2 (one section) -- the
// factorization's sums with them (store_schur).  q has slack entries only, H none but Sigma
// there: no product with H.  Grid ceil(S / CS_N), CS_T threads.  Latencies and the load / store units
// bound it: 5000 scenarios FP32 26 us (warp-per-scenario 22 x 22 solves: 58), FP64 10 scenarios 23 us.
template <int PREC>
__global__ void __launch_bounds__(CS_T, 6) cond_solve_kernel(const Params P, int S, int64_t ld, const BView b,
                                                          const CondFac K, const double* x,
                                                          const double* __restrict__ rc, const double* rz,
                                                          const double* __restrict__ sig,
                                                          const double* __restrict__ hes, bool use_w,
                                                          const int* __restrict__ sing, double* __restrict__ po,
                                                          double* part, int planes) {
    extern __shared__ __align__(16) unsigned char cond_sm[];
    const CondPlace at(S, b);
    const bool live = at.live;
    const int n = at.n, pr = at.pr;
    const int64_t s = at.o;
    if (!__syncthreads_or(live)) return;
    double r[NR], u[NV];
#pragma unroll
    for (int j = 0; j < NR; ++j) r[j] = rc[(int64_t)(NR * n + j) * ld + s];
    cond_solve_prec<PREC>(K, ld, at, r, cond_sm, u);
    if (!live) return;
#pragma unroll
    for (int j = 0; j < NV; ++j) po[(int64_t)(NV * n + j) * ld + s] = u[j];
    if (!planes) return;
    const int sec = stage_sec(n, P.nsec);
    const double qs = slack_q(P, x, ld, sec, b.NP, pr);
    const int64_t o = (int64_t)(NV * n + LS) * ld + s;
    const double a = qs * (rz[o] - sig[o] * u[LS]), c = qs * u[LS];
    if (planes == 2) {
        store_schur(P, sig, hes, use_w, sing, qs, a, c, part, ld, s, n);
    } else {
        const double w[4] = {sec ? a : 0.0, sec ? c : 0.0, sec ? 0.0 : a, sec ? 0.0 : c};
        store_partials<4>(w, part, ld, (int)s, n);
    }
}

// One block-elimination solve after its J^-1 r_c (pv) and Schur step (the steps of the design
// entries in dz's slots): dz = p - q dtheta, g = r_z - (W + Sigma + dw I) dz, dl = J^-T g.  With az,
// al (a correction) they are added to that direction.  g0 (optional): g, for the residual.  r_z and dz
// may be one vector: every entry is read, by the repeated places too (of the same warp), before it
// is written.  Grid
// ceil(S / CS_N), CS_T threads.  5000 scenarios FP32 44-57 us (dz and g, and the
// transposed solve were 13 + 52), the FP64 pipe 42 % busy with the products with H.
template <int PREC>
__global__ void __launch_bounds__(CS_T, 6) cond_direction_kernel(
    const Params P, int S, int64_t ld, const BView b, const CondFac K, const double* __restrict__ hes,
    const double* __restrict__ sig, bool use_w, const double* x, const double* __restrict__ pv,
    const double* rz, double* dzo, double* __restrict__ dlo, double* __restrict__ az,
    double* __restrict__ al, double* __restrict__ g0) {
    extern __shared__ __align__(16) unsigned char cond_sm[];
    const CondPlace at(S, b);
    const bool live = at.live;
    const int n = at.n, pr = at.pr;
    const int64_t s = at.o;
    if (!__syncthreads_or(live)) return;
    const int prc = pr >= 0 ? pr : 0;
    const int sec = stage_sec(n, P.nsec);
    const double dd = dzo[(int64_t)NSC * ld + (int64_t)sec * b.NP + prc], dw = b.ps ? psv(b, PS_DW, prc) : 0.0;
    double g[NV];
    {
        double dz[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) dz[j] = pv[(int64_t)(NV * n + j) * ld + s];
        dz[LS] = fma(-slack_q(P, x, ld, sec, b.NP, prc), dd, dz[LS]);
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            const int64_t o = (int64_t)(NV * n + j) * ld + s;
            g[j] = fma(-(sig[o] + dw), dz[j], rz[o]);
        }
        if (use_w) {
            const double* h = hes + (int64_t)(NHS * n) * ld + s;
#pragma unroll
            for (int i = 0; i < NV; ++i)
#pragma unroll
                for (int j = 0; j <= i; ++j)
                    if (hes_has(i, j)) {
                        const double v = h[(int64_t)c_slotH[i][j] * ld];
                        g[i] = fma(-v, dz[j], g[i]);
                        if (i != j) g[j] = fma(-v, dz[i], g[j]);
                    }
        }
        __syncwarp();
        if (live)
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                const int64_t o = (int64_t)(NV * n + j) * ld + s;
                if (az) az[o] += dz[j];
                else dzo[o] = dz[j];
                if (g0) g0[o] = g[j];
            }
    }
    double dl[NR];
    cond_solve_t_prec<PREC>(K, ld, at, g, cond_sm, dl);
    if (!live) return;
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const int64_t o = (int64_t)(NR * n + j) * ld + s;
        dlo[o] = dl[j];
        if (al) al[o] += dl[j];
    }
}

}  // namespace absorber
