// kernels.cuh -- device kernels of the absorber library (included once, by absorber_lib.cu).
//
// Layout: structure of arrays over scenarios, leading dimension ld (a multiple of 32):
// per-scenario entry v of scenario s lives at [v * ld + s], so a warp touches 32
// consecutive doubles of one entry (one 256-byte coalesced access).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "model.cuh"

namespace absorber {

constexpr int NABV = 11;   // stream-from-above unknowns of stage n+1 read by stage n
constexpr int NBLW = 6;    // stream-from-below unknowns of stage n-1 read by stage n
constexpr int NHS = 66;    // Hessian lower-triangle entries per stage block
constexpr int MAXOWN = 192, MAXABV = 64, MAXBLW = 32;

__host__ __device__ constexpr int abv_var(int a) { return a < 9 ? a : (a == 9 ? LL : LT); }
__host__ __device__ constexpr int blw_var(int b) { return b < 4 ? LY + b : (b == 4 ? LV : LT); }
__host__ __device__ constexpr int stage_type(int n) { return n == 0 ? 0 : (n == N_STAGES - 1 ? 2 : 1); }

struct Ent {
    short slot;        // entry offset inside the stage's CSR segment
    signed char r;     // row inside the stage
    signed char c;     // column: own unknown (0..21), or above index (0..10), or below (0..5)
};

// Pattern tables, identical for every problem (the model is fixed); uploaded once per
// device.  Built on the host by running stage_eval with a recording emitter.
__constant__ short c_slotJ[3][NR][NLOC];
__constant__ int c_segJ[N_STAGES + 1];
__constant__ short c_slotH[NV][NV];
__constant__ Ent c_own[3][MAXOWN];
__constant__ Ent c_hes[NHS];
__constant__ int c_nown[3], c_nabv[3], c_nblw[3];
__constant__ int c_dslot[3];           // the d entry of the stage's hydraulic row
// The stage tables that the factor and solve kernels read with a different entry on
// every lane (a constant-cache read with 32 different addresses is serialized): one
// global-memory copy, which each factor block stages into shared memory.
struct __align__(16) LaneTables {
    Ent own[3][MAXOWN];
    Ent abv[3][MAXABV];
    Ent blw[3][MAXBLW];
    short blwRp[3][NV + 2];        // row pointers of blw (NV + 1 used; padded to 16 bytes)
    short blwCp[3][NV + 2];        // pointers into blwQ by the stage-below unknown fed
    unsigned char blwQ[3][MAXBLW]; // blw entry indices grouped by that unknown (table order)
};
static_assert(sizeof(LaneTables) % 16 == 0, "LaneTables is copied as 16-byte words");
__device__ LaneTables g_lt;
// the Hessian block expanded to both triangles by row (H v)
__constant__ Ent c_hesF[2 * NHS];
__constant__ short c_hesFp[NV + 1];

// bounds of the stage unknowns (10d): lower 0 for fractions, flows and the slack,
// both for T, none for the extents
__host__ __device__ constexpr bool has_lo(int j) { return !(j >= LE && j < LE + 5); }
__host__ __device__ constexpr bool has_hi(int j) { return j == LT; }

// ------------------------------------------------------------------------------------
// problems: a launch covers one or many independent problems (a batch).  Scenario slot
// s belongs to problem pid[s] (-1: padding); per-problem scalars live in device arrays
// ps[field * NP + p].  pid == nullptr means a single problem owning every slot s < S,
// ps == nullptr means no per-problem scalars (every problem active).
// ------------------------------------------------------------------------------------
enum PsField {
    PS_MU = 0,     // barrier parameter
    PS_TAU,        // fraction-to-the-boundary parameter
    PS_ALPHA,      // primal step / trial step
    PS_ALPHAZ,     // bound-multiplier step
    PS_DW,         // primal regularisation delta_w
    PS_ACT,        // 1: problem takes part in this iteration
    PS_LSACT,      // 1: problem takes part in this line-search trial
    PS_SOC,        // 1: the trial follows the second-order-correction direction
    PS_A0,         // coefficient (first trial step) of the SOC right-hand side
    PS_COUNT
};

struct BView {
    const int* pid;
    const double* ps;
    int NP;
};

__device__ inline int prob_of(const BView& b, int s) { return b.pid ? b.pid[s] : 0; }
__device__ inline double psv(const BView& b, int field, int p) { return b.ps[(int64_t)field * b.NP + p]; }
// problem of slot s if it takes part (flag field PS_ACT or PS_LSACT), else -1
__device__ inline int live_prob(const BView& b, int s, int S, int flag) {
    if (s >= S) return -1;
    const int p = prob_of(b, s);
    if (p < 0) return -1;
    if (b.ps && psv(b, flag, p) == 0.0) return -1;
    return p;
}

// ------------------------------------------------------------------------------------
// reductions: every (scenario, stage) thread stores its K partial values at
// part[k * plane + n * ld + s] (plane = N_STAGES * ld); reduce_kernel (vec_kernels.cuh)
// combines them per problem in a fixed order (deterministic)
// ------------------------------------------------------------------------------------
enum RedOp { RSUM = 0, RMAX = 1, RMIN = 2 };

// |a| as an unsigned integer that orders like |a| (the IEEE layout with the sign cleared;
// a NaN orders above +inf): maxima of magnitudes taken on the integer pipe, off the FP64
// pipe, and a NaN among them survives (the key of the maximum is NaN's)
__device__ __forceinline__ unsigned long long mag_key(double a) {
    return (unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ unsigned long long key_max(unsigned long long a, unsigned long long b) {
    return a > b ? a : b;
}
__device__ __forceinline__ double key_double(unsigned long long k) { return __longlong_as_double((long long)k); }
// maximum of magnitude keys over a warp: the high words first, then the low words among the lanes
// that hold the highest
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long key) {
    const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    return ((unsigned long long)mh << 32) | ml;
}

template <int K>
__device__ inline void store_partials(const double (&v)[K], double* part, int64_t ld, int s, int n) {
    const int64_t plane = (int64_t)N_STAGES * ld;
#pragma unroll
    for (int k = 0; k < K; ++k) part[(int64_t)k * plane + (int64_t)n * ld + s] = v[k];
}

// ------------------------------------------------------------------------------------
// A1 + A2: residuals, Jacobian and Lagrangian Hessian values, one thread per
// (scenario, stage); grid (ceil(S / blockDim), N_STAGES).
// ------------------------------------------------------------------------------------
// The evaluation's values in parts of similar length, for threads that compute one part each (PART >= 0):
// four of the residuals, four of the Jacobian, four of the Hessian; PART < 0: everything asked for.  What a
// part leaves out is known at compile time, so the compiler drops what only that needs.
constexpr int EVAL_PARTS = 4;
constexpr int PART_LOG = 3;   // the part of the residuals that also sums the barrier's logarithms
__host__ __device__ constexpr int res_part(int r) {
    return r < 11 || r == R_SX || r == R_SY ? 0 : (r >= R_RX && r < R_RX + 5 ? 1 : (r == R_E ? 2 : 3));
}
__host__ __device__ constexpr int jac_part(int r, int lv) {
    return r < 11 || (r >= R_RX && r < R_RX + 5) ? 0 : (r == R_E ? (lv < NV ? 1 : 2) : 3);
}
__host__ __device__ constexpr int hes_part(int i, int j) {
    return i < 7 ? 0 : (i < LT ? 1 : (j < 9 ? 2 : 3));
}

// PSUM: also the partials |c| summed (by part, added in their order) and maximal (as a key, off the
// FP64 pipe)
template <bool WR, bool WJ, bool WH, bool PSUM, int PART>
struct DevEmit {
    static constexpr bool want_res = WR, want_jac = WJ, want_hes = WH;
    double* cv;
    double* jv;
    double* hv;
    int64_t ld;
    int s, n, t;
    double asum[EVAL_PARTS];
    unsigned long long amax;
    __device__ __forceinline__ void res(int r, double v) {
        if (PART >= 0 && res_part(r) != PART) return;
        if (cv) cv[(int64_t)(NR * n + r) * ld + s] = v;
        if (PSUM) {
            asum[res_part(r)] += fabs(v);
            amax = key_max(amax, mag_key(v));
        }
    }
    __device__ __forceinline__ void jac(int r, int lv, double v) {
        if (PART >= 0 && jac_part(r, lv) != PART) return;
        jv[(int64_t)(c_segJ[n] + c_slotJ[t][r][lv]) * ld + s] = v;
    }
    __device__ __forceinline__ void hes(int i, int j, double v) {
        if (PART >= 0 && hes_part(i, j) != PART) return;
        hv[(int64_t)(NHS * n + c_slotH[i][j]) * ld + s] = v;
    }
};

__device__ inline void load_stage(const Params& P, int S, int64_t ld, const double* __restrict__ x,
                                  const double* __restrict__ dx, double alpha, const double* __restrict__ feed,
                                  int s, int n, int p, int NP, StageIn& in) {
    const double* xs = x + s;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        double v = xs[(int64_t)(NV * n + j) * ld];
        if (dx) v += alpha * dx[(int64_t)(NV * n + j) * ld + s];
        in.q[j] = v;
    }
    in.has_above = n + 1 < N_STAGES;
    in.has_below = n > 0;
    if (in.has_above) {
#pragma unroll
        for (int a = 0; a < NABV; ++a) {
            const int64_t o = (int64_t)(NV * (n + 1) + abv_var(a)) * ld + s;
            double v = x[o];
            if (dx) v += alpha * dx[o];
            in.qa[a] = a < 9 ? mul_rn(P.sx[a], v) : (a == 9 ? v : mul_rn(P.sT, v));
        }
    } else {
#pragma unroll
        for (int l = 0; l < 9; ++l) in.qa[l] = feed[(int64_t)(F_XIN + l) * ld + s];
        in.qa[9] = feed[(int64_t)F_LIN * ld + s];
        in.qa[10] = feed[(int64_t)F_TIN * ld + s];
    }
    if (in.has_below) {
#pragma unroll
        for (int b = 0; b < NBLW; ++b) {
            const int64_t o = (int64_t)(NV * (n - 1) + blw_var(b)) * ld + s;
            double v = x[o];
            if (dx) v += alpha * dx[o];
            in.qb[b] = b < 4 ? mul_rn(P.sy[b], v) : (b == 4 ? v : mul_rn(P.sT, v));
        }
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) in.qb[j] = feed[(int64_t)(F_Y0 + j) * ld + s];
        in.qb[4] = feed[(int64_t)F_V0 * ld + s];
        in.qb[5] = feed[(int64_t)F_T0 * ld + s];
    }
    const int64_t od = (int64_t)NSC * ld + (int64_t)stage_sec(n, P.nsec) * NP + p;   // its section's diameter
    in.d = x[od] + (dx ? alpha * dx[od] : 0.0);
    in.P = stage_pres(P, feed[(int64_t)F_P * ld + s], n);
}

// The evaluation's argument list: at x (trial = false: the problems flagged PS_ACT) or at x + alpha_p dir
// (trial = true: those flagged PS_LSACT; dir = dxB where PS_SOC is set, else dxA).
struct EvalArgs {
    int S;
    int64_t ld;
    BView b;
    bool trial;
    const double *x, *dxA, *dxB, *lam, *feed;
    double *c, *jac, *hes;
    double* part;
};

// what scenario slot s and stage n ask for; false: the slot takes no part.  PSUM: v = |c| summed over the
// part's rows, their max, the sum of the barrier logs of the stage unknowns.
template <bool WR, bool WJ, bool WH, bool PSUM, int PART>
__device__ __forceinline__ bool eval_body(const Params& P, const EvalArgs& A, int s, int n, double (&v)[3]) {
    const int64_t ld = A.ld;
    const int p = live_prob(A.b, s, A.S, A.trial ? PS_LSACT : PS_ACT);
    if (p < 0) return false;
    DevEmit<WR, WJ, WH, PSUM, PART> em;
    em.cv = A.c;
    em.jv = A.jac;
    em.hv = A.hes;
    em.ld = ld;
    em.s = s;
    em.n = n;
    em.t = stage_type(n);
#pragma unroll
    for (int k = 0; k < EVAL_PARTS; ++k) em.asum[k] = 0.0;
    em.amax = 0;
    StageIn in;
    const double* dx = nullptr;
    double alpha = 0.0;
    if (A.trial) {
        dx = (A.b.ps && psv(A.b, PS_SOC, p) != 0.0) ? A.dxB : A.dxA;
        alpha = psv(A.b, PS_ALPHA, p);
    }
    load_stage(P, A.S, ld, A.x, dx, alpha, A.feed, s, n, p, A.b.NP, in);
    StageLam L;
    if (WH) {
        const double* lam = A.lam;
#pragma unroll
        for (int r = 0; r < NR; ++r) L.own[r] = lam[(int64_t)(NR * n + r) * ld + s];
        if (n > 0) {
#pragma unroll
            for (int k = 0; k < 9; ++k) L.below[k] = lam[(int64_t)(NR * (n - 1) + k) * ld + s];
            L.below[9] = lam[(int64_t)(NR * (n - 1) + R_E) * ld + s];
        }
        if (n + 1 < N_STAGES) {
#pragma unroll
            for (int k = 0; k < 4; ++k) L.above[k] = lam[(int64_t)(NR * (n + 1) + 7 + k) * ld + s];
            L.above[4] = lam[(int64_t)(NR * (n + 1) + R_E) * ld + s];
        }
    }
    stage_eval(P, in, WH ? &L : nullptr, em);
    if (WH && n == 0 && (PART < 0 || PART == EVAL_PARTS - 1)) {
        // the scenario's share of d-d: -u_max pi / 2 * sum_n lambda_hydraulic, one entry per
        // section (its stages' rows)
        for (int k = 0; k < P.nsec; ++k) {
            double sl = 0.0;
#pragma unroll
            for (int m = 0; m < N_STAGES; ++m)
                if (stage_sec(m, P.nsec) == k) sl += A.lam[(int64_t)(NR * m + R_H) * ld + s];
            A.hes[(int64_t)(NHS * N_STAGES + k) * ld + s] = -P.u_max * M_PI * 0.5 * sl;
        }
    }
    if (PSUM) {
        v[0] = PART >= 0 ? em.asum[PART < 0 ? 0 : PART] : ((em.asum[0] + em.asum[1]) + em.asum[2]) + em.asum[3];
        v[1] = key_double(em.amax);
        v[2] = 0.0;
    }
    if (PSUM && (PART < 0 || PART == PART_LOG)) {
        // sum of ln(slack) over the stage's 18 bounds as the logarithm of their product: the
        // product is carried as a mantissa in [1, 2) times a power of two (exponent read from
        // the bit pattern), so it neither overflows nor underflows; a slack that is not
        // positive and finite makes the sum NaN (the trial is rejected as before)
        double m = 1.0;
        long long e2 = 0;
        bool bad = false;
        auto take = [&](double sl) {
            // positive and finite: a bit pattern in [1, that of +inf)
            bad = bad || (unsigned long long)__double_as_longlong(sl) - 1ull >= (0x7ffull << 52) - 1ull;
            m *= sl;
            const unsigned long long bits = (unsigned long long)__double_as_longlong(m);
            const int ex = (int)((bits >> 52) & 0x7ffull);
            if (ex == 0 || ex == 0x7ff) {
                bad = true;
                return;
            }
            e2 += ex - 1023;
            m = __longlong_as_double((long long)((bits & ~(0x7ffull << 52)) | (1023ull << 52)));
        };
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            if (has_lo(j)) take(in.q[j] - (j == LT ? P.Tlo_s : 0.0));
            if (has_hi(j)) take(P.Thi_s - in.q[j]);
        }
        v[2] = bad ? NAN : fma((double)e2, 0.69314718055994530942, ln_tab(m));   // ln 2
    }
    return true;
}

// One thread per (scenario, stage), in 32-thread blocks: FP64 instructions bound it (5000 scenarios, all
// values: 121 us; residuals only 45 us), and 1570 blocks at 5000 scenarios share
// out evenly over 152 SMs.
constexpr int EVAL_T = 32;
template <bool WR, bool WJ, bool WH, bool PSUM>
__global__ void __launch_bounds__(EVAL_T) eval_kernel(const Params P, const EvalArgs A) {
    const int s = blockIdx.x * EVAL_T + threadIdx.x, n = blockIdx.y;
    double v[3];
    if (eval_body<WR, WJ, WH, PSUM, -1>(P, A, s, n, v) && PSUM) store_partials<3>(v, A.part, A.ld, s, n);
}

// the part of a warp of eval_split_kernel
template <bool WR, bool WJ, bool WH, bool PSUM>
__device__ __forceinline__ bool eval_part(const Params& P, const EvalArgs& A, int part, int s, int n, double (&v)[3]) {
    if (part == 0) return eval_body<WR, WJ, WH, PSUM, 0>(P, A, s, n, v);
    if (part == 1) return eval_body<WR, WJ, WH, PSUM, 1>(P, A, s, n, v);
    if (part == 2) return eval_body<WR, WJ, WH, PSUM, 2>(P, A, s, n, v);
    return eval_body<WR, WJ, WH, PSUM, 3>(P, A, s, n, v);
}

// The same by four warps per 32 (scenario, stage) pairs, each a part, in blocks of their own for the
// residuals, the Jacobian and the Hessian -- what: 0, 1, 2, a digit per blockIdx.z -- for sizes at which
// the threads of eval_kernel leave schedulers idle: a warp alone on its scheduler issues an FP64
// instruction per 64 cycles whatever else the SM does, so twelve short threads finish sooner though
// together they compute more.  Values and partials are eval_kernel's bit for bit (model.cuh), so a
// problem's do not depend on the batch it runs in.
template <bool PSUM>
__global__ void __launch_bounds__(EVAL_PARTS * EVAL_T) eval_split_kernel(const Params P, const EvalArgs A, int what) {
    __shared__ double sh[3][EVAL_PARTS][EVAL_T];
    const int lane = threadIdx.x, part = threadIdx.y;
    const int s = blockIdx.x * EVAL_T + lane, n = blockIdx.y;
    const int kind = (what >> (4 * blockIdx.z)) & 15;
    double v[3];
    if (kind == 1) {
        eval_part<false, true, false, false>(P, A, part, s, n, v);
    } else if (kind == 2) {
        eval_part<false, false, true, false>(P, A, part, s, n, v);
    } else {
        const bool live = eval_part<true, false, false, PSUM>(P, A, part, s, n, v);
        if (PSUM) {
#pragma unroll
            for (int k = 0; k < 3; ++k) sh[k][part][lane] = live ? v[k] : 0.0;
            __syncthreads();
            if (part == 0 && live) {
                unsigned long long mx = 0;
                v[0] = ((sh[0][0][lane] + sh[0][1][lane]) + sh[0][2][lane]) + sh[0][3][lane];
#pragma unroll
                for (int q = 0; q < EVAL_PARTS; ++q) {
                    mx = key_max(mx, mag_key(sh[1][q][lane]));
                }
                v[1] = key_double(mx);
                v[2] = sh[2][PART_LOG][lane];
                store_partials<3>(v, A.part, A.ld, s, n);
            }
        }
    }
}

// the stage pattern at compile time: Jacobian entries of a stage's own unknowns, and Hessian entries
// (lower triangle)
__host__ __device__ constexpr bool own_has(int r, int c) {
    if (r < 11) {
        if (r < 9 && (c == r || c == LL)) return true;
        if (r >= 7 && (c == LY + r - 7 || c == LV)) return true;
        return c >= LE && c < LE + 5 && nu(r, c - LE) != 0;
    }
    if (r == R_VH) return c == LY + 1 || c == 8 || c == LT;
    if (r == R_VC) return c == LY || c == LT || (c < 9 && in_henry(c));
    if (r >= R_RX && r < R_RX + 5) return c == LT || (c < 9 && nu(c, r - R_RX) != 0);
    if (r == R_SX) return c < 9;
    if (r == R_SY) return c >= LY && c < LY + 4;
    if (r == R_E) return c <= LT;
    return c == LV || c == LT || c == LS;
}
// row r reads the stage above's unknown a (of the 11) / the stage below's b (of the 6)
__host__ __device__ constexpr bool abv_has(int r, int a) { return r == R_E || (r < 9 && (a == r || a == 9)); }
__host__ __device__ constexpr bool blw_has(int r, int b) {
    return r == R_E || (r >= 7 && r < 11 && (b == r - 7 || b == 4));
}
__host__ __device__ constexpr bool hes_has(int i, int j) {
    if (i < 9) return j <= i && ((in_henry(i) && in_henry(j)) || i == j);
    if (i == LL) return j < 9;
    if (i == LV) return j >= LY && j < LY + 4;
    return i == LT && j <= LT;
}

// The products J v and J^T y of a stage shared out over four warps, with 150 entries each: rows and
// unknowns grouped so that every warp has 70 to 80 of the 300 multiply-adds, all of it unrolled code
// at fixed places (no tables, no loops).
constexpr int NGRP = 4;
__host__ __device__ constexpr int row_grp(int r) {
    return r == R_E || r == R_VH || r == R_SY ? 0 : (r == R_SX || r == R_VC || r == 7 || r == 8 ? 1 : (r < 7 ? 2 : 3));
}
__host__ __device__ constexpr int col_grp(int j) {
    return j == LL || j == LV ? 0 : (j < 5 ? 1 : (j < 9 || j == LE || j == LE + 1 ? 2 : 3));
}

// where a (scenario, stage)'s Jacobian entries lie: its own stage's and its neighbours' segments
struct StageJac {
    const double *own, *below, *above;   // segments of stage n, n - 1, n + 1 at the scenario
    int t, tb, ta;                       // their stage types
    int64_t ld;
    __device__ __forceinline__ StageJac(const double* __restrict__ jac, int64_t ld_, int s, int n) : ld(ld_) {
        t = stage_type(n);
        tb = n > 0 ? stage_type(n - 1) : 0;
        ta = n + 1 < N_STAGES ? stage_type(n + 1) : 0;
        own = jac + (int64_t)c_segJ[n] * ld + s;
        below = jac + (int64_t)c_segJ[n > 0 ? n - 1 : 0] * ld + s;
        above = jac + (int64_t)c_segJ[n + 1 < N_STAGES ? n + 1 : 0] * ld + s;
    }
    __device__ __forceinline__ double at(int r, int lv) const { return own[(int64_t)c_slotJ[t][r][lv] * ld]; }
    __device__ __forceinline__ double at_below(int r, int lv) const { return below[(int64_t)c_slotJ[tb][r][lv] * ld]; }
    __device__ __forceinline__ double at_above(int r, int lv) const { return above[(int64_t)c_slotJ[ta][r][lv] * ld]; }
};

// f(0), f(1), ... f(N - 1) with compile-time arguments
template <int I, int N, class F>
__device__ __forceinline__ void static_for(const F& f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, N>(f);
    }
}

// a <- a + sgn (J^T y)_j for unknown j of stage n; y a row vector
template <int SGN, int j>
__device__ __forceinline__ double jt_col(const StageJac& J, const double* __restrict__ y, int s, int n, double a) {
    const double* yn = y + (int64_t)(NR * n) * J.ld + s;
    static_for<0, NR>([&](auto R) {
        constexpr int r = decltype(R)::value;
        if constexpr (own_has(r, j)) a = fma(SGN * J.at(r, j), yn[(int64_t)r * J.ld], a);
    });
    static_for<0, NABV>([&](auto K) {
        constexpr int k = decltype(K)::value;
        if constexpr (abv_var(k) == j) {
            if (n > 0) {
                const double* yb = yn - (int64_t)NR * J.ld;
                static_for<0, NR>([&](auto R) {
                    constexpr int r = decltype(R)::value;
                    if constexpr (abv_has(r, k)) a = fma(SGN * J.at_below(r, AX + k), yb[(int64_t)r * J.ld], a);
                });
            }
        }
    });
    static_for<0, NBLW>([&](auto K) {
        constexpr int k = decltype(K)::value;
        if constexpr (blw_var(k) == j) {
            if (n + 1 < N_STAGES) {
                const double* ya = yn + (int64_t)NR * J.ld;
                static_for<0, NR>([&](auto R) {
                    constexpr int r = decltype(R)::value;
                    if constexpr (blw_has(r, k)) a = fma(SGN * J.at_above(r, BY + k), ya[(int64_t)r * J.ld], a);
                });
            }
        }
    });
    return a;
}

// a <- a - (J v)_r for row r of stage n; v a primal vector, vd the step of its section's diameter
template <int r>
__device__ __forceinline__ double jv_row(const StageJac& J, const double* __restrict__ v, double vd, int s, int n,
                                         double a) {
    const double* vn = v + (int64_t)(NV * n) * J.ld + s;
    static_for<0, NV>([&](auto C) {
        constexpr int j = decltype(C)::value;
        if constexpr (own_has(r, j)) a = fma(-J.at(r, j), vn[(int64_t)j * J.ld], a);
    });
    if (n + 1 < N_STAGES)
        static_for<0, NABV>([&](auto K) {
            constexpr int k = decltype(K)::value;
            if constexpr (abv_has(r, k)) a = fma(-J.at(r, AX + k), vn[(int64_t)(NV + abv_var(k)) * J.ld], a);
        });
    if (n > 0)
        static_for<0, NBLW>([&](auto K) {
            constexpr int k = decltype(K)::value;
            if constexpr (blw_has(r, k)) a = fma(-J.at(r, BY + k), vn[(int64_t)(blw_var(k) - NV) * J.ld], a);
        });
    if constexpr (r == R_H) a = fma(-J.own[(int64_t)c_dslot[J.t] * J.ld], vd, a);
    return a;
}

// ------------------------------------------------------------------------------------
// sparse products with the stage-structured Jacobian / Hessian
// ------------------------------------------------------------------------------------
// ((W + Sigma + dw I) v)_j for unknown j of stage n (W block diagonal by stage);
// use_w = false gives (Sigma + dw I) v
__device__ __forceinline__ double hv_one(int64_t ld, const double* __restrict__ hes, const double* __restrict__ sig,
                                double dw, bool use_w, const double* __restrict__ v, int s, int n, int j) {
    const int64_t o = (int64_t)(NV * n + j) * ld + s;
    double a = (sig[o] + dw) * v[o];
    if (use_w)
        for (int k = c_hesFp[j]; k < c_hesFp[j + 1]; ++k) {
            const Ent e = c_hesF[k];
            a += hes[(int64_t)(NHS * n + e.slot) * ld + s] * v[(int64_t)(NV * n + e.c) * ld + s];
        }
    return a;
}

}  // namespace absorber
