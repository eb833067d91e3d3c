// kernels_warp.cuh -- warp-cooperative factors and solves of the uncondensed 22 x 22 stage
// blocks: the solves of the tensor-core FP32 factor (factor_gj_tc_kernel, kernels_tc.cuh), which
// keeps stage-block inverses, and the FP64 block LU with partial pivoting
// (factor_lu_kernel) with its solves.  Both read every Jacobian value: they serve, besides
// ABS_PREC_FP32_TC, the Jacobians that the condensed factors do not cover (kernels_cond.cuh:
// rows scaled or values edited after the evaluation).
//
// One warp per scenario; vectors live one entry per lane, broadcasts are warp shuffles.
// factor_lu_kernel keeps a stage block in shared memory while the warp works on it: pivot
// search with rows on lanes, the trailing update with columns on lanes, the super-diagonal
// block B_n appended as 11 extra columns, so that the elimination yields L^-1 P B_n, then
// U G_n = L^-1 P B_n by backward substitution.  FP64 latency bounds it (20000 scenarios 8.9 ms):
// the condensed factors are 13 times as fast where they apply.
// Factor storage is per scenario and contiguous (internal layout, not part of the C ABI): the
// inverse or LU [s][n][22][22] (the reciprocals of the pivots on U's diagonal), G[s][n][22][11]
// and the row order piv[s][n][22][2] (see PIV_BYTES), so every warp access to the factors is
// coalesced.
#pragma once

#include <type_traits>

#include "kernels.cuh"

namespace absorber {

constexpr int NCA = NV + NABV;    // augmented columns [A_n | B_n]
constexpr int PADA = NCA + 1;     // shared-memory row stride of the augmented block
constexpr int PADL = NV + 1;      // shared-memory row stride of a staged LU block
constexpr int WPB_F = 4;          // default warps (scenarios) per block, factor
constexpr int WPB_S = 4;          // default warps (scenarios) per block, solves

__host__ __device__ constexpr int64_t lu_off(int64_t s, int n) { return (s * N_STAGES + n) * (int64_t)(NV * NV); }
__host__ __device__ constexpr int64_t g_off(int64_t s, int n) { return (s * N_STAGES + n) * (int64_t)(NV * NABV); }
// row order of a factored stage block: (perm[i], ipos[i]) byte pairs for i < 22, perm[i]
// the block row at position i of P A = L U and ipos[j] the position of block row j
constexpr int PIV_BYTES = 2 * NV;
__host__ __device__ constexpr int64_t pv_off(int64_t s, int n) { return (s * N_STAGES + n) * (int64_t)PIV_BYTES; }

template <class T>
__device__ inline T shfl(T v, int src) {
    return __shfl_sync(0xffffffffu, v, src);
}

// FP32 pivot key: |a| with its 5 lowest mantissa bits replaced by 31 - position, so that
// one warp maximum both finds the pivot and breaks ties: the candidate of largest |a| up
// to a relative 2^-18, the lowest position among those (threshold partial pivoting; an
// all-zero column takes its lowest position, a NaN always wins)
__device__ __forceinline__ unsigned pivot_key32(float a, int pos) {
    return (__float_as_uint(a) & 0x7fffffe0u) | (unsigned)(31 - pos);
}
__device__ __forceinline__ int key_position(unsigned key) { return 31 - (int)(key & 31u); }

__device__ inline float recip(float a) { return 1.0f / a; }
// FP32 seed and two Newton steps r <- r (2 - a r) (|a| in the normal FP32 range; division otherwise)
__device__ inline double recip(double a) {
    const double m = fabs(a);
    if (m > 1e-30 && m < 1e30) {
        double r = (double)(1.0f / (float)a);
        r = r * fma(-a, r, 2.0);
        r = r * fma(-a, r, 2.0);
        return r;
    }
    return 1.0 / a;
}

// the per-lane stage tables, copied once per block into shared memory (every thread of
// the block takes part; call before any warp leaves)
__device__ inline void stage_lane_tables(LaneTables& lt) {
    const int4* src = reinterpret_cast<const int4*>(&g_lt);
    int4* dst = reinterpret_cast<int4*>(&lt);
    constexpr int NW = (int)(sizeof(LaneTables) / sizeof(int4));
    for (int i = threadIdx.x; i < NW; i += blockDim.x) dst[i] = src[i];
    __syncthreads();
}

constexpr int OWN_PER_LANE = MAXOWN / 32, ABV_PER_LANE = MAXABV / 32;

// the Jacobian values of stage n's own and super-diagonal entries that lane `lane`
// scatters (entries lane, lane + 32, ...), every load issued before the first use
struct StageLoads {
    Ent eo[OWN_PER_LANE];
    double vo[OWN_PER_LANE];
    Ent ea[ABV_PER_LANE];
    double va[ABV_PER_LANE];
    int no, na;
    __device__ inline void fetch(const LaneTables& lt, int n, int64_t ld, int s, int lane,
                                 const double* __restrict__ jac) {
        const int t = stage_type(n);
        const int base = c_segJ[n];
        no = c_nown[t];
        na = n + 1 < N_STAGES ? c_nabv[t] : 0;
#pragma unroll
        for (int i = 0; i < OWN_PER_LANE; ++i) {
            const int k = lane + 32 * i;
            eo[i] = lt.own[t][k < no ? k : 0];
        }
#pragma unroll
        for (int i = 0; i < ABV_PER_LANE; ++i) {
            const int k = lane + 32 * i;
            ea[i] = lt.abv[t][k < na ? k : 0];
        }
#pragma unroll
        for (int i = 0; i < OWN_PER_LANE; ++i)
            vo[i] = lane + 32 * i < no ? jac[(int64_t)(base + eo[i].slot) * ld + s] : 0.0;
#pragma unroll
        for (int i = 0; i < ABV_PER_LANE; ++i)
            va[i] = lane + 32 * i < na ? jac[(int64_t)(base + ea[i].slot) * ld + s] : 0.0;
    }
    // scatter into the augmented block (row stride P, B_n from column NV)
    template <class T, int P>
    __device__ inline void scatter(T* A, int lane) const {
#pragma unroll
        for (int i = 0; i < OWN_PER_LANE; ++i)
            if (lane + 32 * i < no) A[eo[i].r * P + eo[i].c] = (T)vo[i];
#pragma unroll
        for (int i = 0; i < ABV_PER_LANE; ++i)
            if (lane + 32 * i < na) A[ea[i].r * P + NV + ea[i].c] = (T)va[i];
    }
};

constexpr int NPR = (NCA + 1) / 2;   // float pairs of [A_n | B_n] per row (column 33: padding)
constexpr int NBLWV = 6;             // unknowns of the stage below in a row's coupling (C_n)
constexpr int PADQ = 36;             // assembly row stride (rows 16-byte aligned)
constexpr int UINV = 36;             // broadcast buffer: the pivot's reciprocal

__device__ __forceinline__ float& rv(float2* r, int j) { return (j & 1) ? r[j >> 1].y : r[j >> 1].x; }

// ---- FP64 block LU ----
// a stage's LU block and row order fetched into registers ahead of use (the next
// stage's loads overlap the current stage's work), then committed: the block to shared
// memory, lane i's (perm[i], ipos[i]) to registers (lanes >= 22: i itself)
constexpr int LU_PER_LANE = (NV * NV + 31) / 32;
struct LUPrefetch {
    double v[LU_PER_LANE];
    uchar2 p;
    __device__ inline void fetch(const double* __restrict__ LU, const unsigned char* __restrict__ piv, int64_t s, int n,
                                 int lane) {
        const double* src = LU + lu_off(s, n);
#pragma unroll
        for (int i = 0; i < LU_PER_LANE; ++i) {
            const int e = lane + 32 * i;
            v[i] = e < NV * NV ? src[e] : 0.0;
        }
        p = lane < NV ? reinterpret_cast<const uchar2*>(piv + pv_off(s, n))[lane]
                      : make_uchar2((unsigned char)lane, (unsigned char)lane);
    }
    __device__ inline void commit(double (*A)[PADL], int& perm, int& ipos, int lane) const {
#pragma unroll
        for (int i = 0; i < LU_PER_LANE; ++i) {
            const int e = lane + 32 * i;
            if (e < NV * NV) A[e / NV][e % NV] = v[i];
        }
        perm = p.x;
        ipos = p.y;
    }
};

// assemble stage n's augmented block [A_n | B_n] of scenario s in shared memory (own
// entries, the super-diagonal coupling B_n, the Schur update A_n -= C_n G_{n-1}) and
// return the threshold below which a pivot marks the block singular
__device__ inline double assemble_stage(int n, int64_t ld, int s, int lane, const double* __restrict__ jac, double pivtol,
                                   const LaneTables& lt, double (*A)[PADA], const double (*Gp)[NABV]) {
    const int t = stage_type(n);
    const int base = c_segJ[n];
    StageLoads L;
    L.fetch(lt, n, ld, s, lane, jac);
    const int nq = n > 0 ? c_nblw[t] : 0;
    const double cvq = lane < nq ? jac[(int64_t)(base + lt.blw[t][lane].slot) * ld + s] : 0.0;   // entry q on lane q
    for (int e = lane; e < NV * NCA; e += 32) A[e / NCA][e % NCA] = 0.0;
    __syncwarp();
    L.scatter<double, PADA>(&A[0][0], lane);
    __syncwarp();
    // Schur update with the previous stage: A_n -= C_n G_{n-1}
    for (int k = 0; k < nq; ++k) {
        const Ent e = lt.blw[t][k];
        const double cv = shfl(cvq, k);
        if (lane < NABV) A[e.r][abv_var(lane)] = fma(-cv, Gp[blw_var(e.c)][lane], A[e.r][abv_var(lane)]);
        __syncwarp();
    }
    // largest entry of the block (for the singularity test)
    unsigned long long kmax = 0ull;
    for (int e = lane; e < NV * NV; e += 32) {
        kmax = key_max(kmax, mag_key(A[e / NV][e % NV]));
    }
    kmax = warp_max_key(kmax);
    return pivtol * key_double(kmax);
}

// LU factors, row order and G of every active scenario; sing[s] = 1 where a pivot is below pivtol of
// its block's largest entry (replaced by that bound)
template <int WPB = WPB_F>
__global__ void __launch_bounds__(32 * WPB) factor_lu_kernel(int S, int64_t ld, const BView b,
                                                                 const double* __restrict__ jac, double* __restrict__ LU,
                                                                 unsigned char* __restrict__ piv, double* __restrict__ G,
                                                                 int* __restrict__ sing, double pivtol) {
    __shared__ double sA[WPB][NV][PADA];
    __shared__ double sG[WPB][NV][NABV];
    __shared__ LaneTables lt;
    stage_lane_tables(lt);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = blockIdx.x * WPB + warp;
    // whole warps leave together; no block-level barriers below
    if (live_prob(b, s, S, PS_ACT) < 0) return;
    double(*A)[PADA] = sA[warp];
    double(*Gp)[NABV] = sG[warp];
    int singular = 0;
    for (int n = 0; n < N_STAGES; ++n) {
        const double tiny = assemble_stage(n, ld, s, lane, jac, pivtol, lt, A, Gp);
        const unsigned long long ktiny = mag_key(tiny);
        unsigned char* pv = piv + pv_off(s, n);
        int orig = lane;   // block row now at position lane
        // LU with partial pivoting, row operations on all 33 columns, fully unrolled (static
        // shared-memory offsets, independent row updates)
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            // the largest |value| among the rows left, ties to the lowest row
            const bool cand = lane >= k && lane < NV;
            const unsigned long long key = cand ? mag_key(A[lane][k]) : 0ull, kbest = warp_max_key(key);
            int p = __ffs((int)__ballot_sync(0xffffffffu, cand && key == kbest)) - 1;
            if (p < 0 || p >= NV) p = k;
            if (p != k) {
                for (int j = lane; j < NCA; j += 32) {
                    const double a = A[k][j];
                    A[k][j] = A[p][j];
                    A[p][j] = a;
                }
                const int ok = __shfl_sync(0xffffffffu, orig, k), op = __shfl_sync(0xffffffffu, orig, p);
                if (lane == k) orig = op;
                if (lane == p) orig = ok;
            }
            __syncwarp();
            double ukk = A[k][k];
            if (!(mag_key(ukk) > ktiny) || ukk != ukk) {
                singular = 1;
                ukk = (ukk < 0.0 ? -1.0 : 1.0) * (tiny > 0.0 ? tiny : 1.0);
            }
            const double inv = recip(ukk);
            if (lane > k && lane < NV) A[lane][k] *= inv;
            __syncwarp();
            const int j = k + 1 + lane;
            if (j < NCA) {
                const double akj = A[k][j];
#pragma unroll
                for (int i = k + 1; i < NV; ++i) A[i][j] = fma(-A[i][k], akj, A[i][j]);
            }
            if (lane == 0) A[k][k] = inv;
            __syncwarp();
        }
        // U G = L^-1 P B: lanes 0..21 = (column a = lane % 11, row parity lane / 11)
        if (n + 1 < N_STAGES) {
            const int a = lane % NABV, grp = lane / NABV;
#pragma unroll
            for (int i = NV - 1; i >= 0; --i) {
                const double g = A[i][NV + a] * A[i][i];
                __syncwarp();
                if (grp < 2) {
#pragma unroll
                    for (int r = grp; r < i; r += 2) A[r][NV + a] = fma(-A[r][i], g, A[r][NV + a]);
                    if (grp == 0) A[i][NV + a] = g;
                }
                __syncwarp();
            }
            double* Gn = G + g_off(s, n);
            for (int e = lane; e < NV * NABV; e += 32) {
                const double g = A[e / NABV][NV + e % NABV];
                Gn[e] = g;
                Gp[e / NABV][e % NABV] = g;
            }
        }
        double* Ln = LU + lu_off(s, n);
        for (int e = lane; e < NV * NV; e += 32) Ln[e] = A[e / NV][e % NV];
        if (lane < NV) {
            pv[2 * lane] = (unsigned char)orig;
            pv[2 * orig + 1] = (unsigned char)lane;
        }
        __syncwarp();
    }
    if (lane == 0) sing[s] = singular;
}

// w <- At^-1 w, lane i holding w_i (lanes >= 22 carry zeros): P w in one shuffle, then
// L forward and U backward (unrolled: the loads of A run ahead of the shuffle chain)
__device__ inline double lu_apply_warp(const double (*A)[PADL], int perm, int lane, double w) {
    w = shfl(w, perm);
#pragma unroll
    for (int k = 0; k < NV - 1; ++k) {
        const double wk = shfl(w, k);
        if (lane > k && lane < NV) w -= A[lane][k] * wk;
    }
#pragma unroll
    for (int k = NV - 1; k >= 0; --k) {
        if (lane == k) w *= A[k][k];
        const double wk = shfl(w, k);
        if (lane < k) w -= A[lane][k] * wk;
    }
    return w;
}

// w <- At^-T w:  U^T forward, L^T backward, then P^T w in one shuffle
__device__ inline double lu_apply_t_warp(const double (*A)[PADL], int ipos, int lane, double w) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        if (lane == k) w *= A[k][k];
        const double wk = shfl(w, k);
        if (lane > k && lane < NV) w -= A[k][lane] * wk;
    }
#pragma unroll
    for (int k = NV - 1; k > 0; --k) {
        const double wk = shfl(w, k);
        if (lane < k) w -= A[k][lane] * wk;
    }
    return shfl(w, ipos);
}

// ---- stage-block inverses (FP32) ----
// Lane i's row i of the stage-block inverse M (columns in
// position order) and its row-order pair, fetched a stage ahead.  The block solve
// y = A_n^-1 w is y_i = sum_c M_ic w_perm[c] (two interleaved accumulations: even and odd c)
constexpr int NPI = NV / 2;
struct InvRowFetch {
    float2 a[NPI];
    uchar2 p;
    __device__ inline void fetch(const float* __restrict__ AI, const unsigned char* __restrict__ piv, int64_t s,
                                 int n, int lane) {
        const float2* src = reinterpret_cast<const float2*>(AI + lu_off(s, n) + (lane < NV ? lane : 0) * NV);
#pragma unroll
        for (int m = 0; m < NPI; ++m) a[m] = lane < NV ? src[m] : make_float2(0.f, 0.f);
        p = lane < NV ? reinterpret_cast<const uchar2*>(piv + pv_off(s, n))[lane]
                      : make_uchar2((unsigned char)lane, (unsigned char)lane);
    }
    __device__ inline float apply(float w) const {
        w = shfl(w, (int)p.x);
        float e = 0.f, o = 0.f;
#pragma unroll
        for (int m = 0; m < NPI; ++m) {
            e = fmaf(a[m].x, shfl(w, 2 * m), e);
            o = fmaf(a[m].y, shfl(w, 2 * m + 1), o);
        }
        return e + o;
    }
};
// ... and lane c's column c, for the transposed block solve: u_c = sum_i M_ic w_i, then
// v_j = u_ipos[j]
struct InvColFetch {
    float c[NV];
    uchar2 p;
    __device__ inline void fetch(const float* __restrict__ AI, const unsigned char* __restrict__ piv, int64_t s,
                                 int n, int lane) {
        const float* src = AI + lu_off(s, n) + (lane < NV ? lane : 0);
#pragma unroll
        for (int i = 0; i < NV; ++i) c[i] = lane < NV ? src[i * NV] : 0.f;
        p = lane < NV ? reinterpret_cast<const uchar2*>(piv + pv_off(s, n))[lane]
                      : make_uchar2((unsigned char)lane, (unsigned char)lane);
    }
    __device__ inline float apply(float w) const {
        float e = 0.f, o = 0.f;
#pragma unroll
        for (int i = 0; i < NV; i += 2) {
            e = fmaf(c[i], shfl(w, i), e);
            o = fmaf(c[i + 1], shfl(w, i + 1), o);
        }
        return shfl(e + o, (int)p.y);
    }
};

// the coupling of stage n to the stage below (C_n: entry q on lane q), fetched a stage
// ahead of use: the entry's Jacobian value (kept in double until used, so that the load
// does not stall the fetch), the stage-below unknown it multiplies (row solves) or its
// row (transposed solves), and lane j's group of entries -- those of row j (row solves)
// or those feeding stage-below unknown j (transposed solves), in table order
constexpr int NBLWC = 8;   // entries feeding one stage-below unknown, at most
struct CouplingFetch {
    double cv;
    int src, q0, nb;
    unsigned char qi[NBLWC];   // transposed solves: the group's entry indices
    template <bool TRANS>
    __device__ inline void fetch(int n, int64_t ld, int s, int lane, const double* __restrict__ jac) {
        const int t = stage_type(n), base = c_segJ[n], nq = c_nblw[t];
        const Ent e = g_lt.blw[t][lane < nq ? lane : 0];
        cv = lane < nq ? jac[(int64_t)(base + e.slot) * ld + s] : 0.0;
        src = lane < nq ? (TRANS ? (int)e.r : blw_var(e.c)) : 0;
        const short* ptr = TRANS ? g_lt.blwCp[t] : g_lt.blwRp[t];
        q0 = lane < NV ? ptr[lane] : 0;
        nb = lane < NV ? ptr[lane + 1] - q0 : 0;
        if (TRANS) {
#pragma unroll
            for (int i = 0; i < NBLWC; ++i) qi[i] = g_lt.blwQ[t][i < nb ? q0 + i : 0];
        }
    }
};

// J_s x = r (NRHS right-hand sides; a null r[k] means b = dc/dtheta_bsec, the border
// column of design entry bsec: nonzero in the hydraulic rows of that section's stages),
// one warp per scenario.
// T = float: LU holds the stage-block inverses and each block solve is a matrix-vector product;
// double: LU factors, staged in the warp's shared-memory block A.  The block solves of scenario s
// (problem pr) by its warp.
template <class T, int NRHS>
__device__ __forceinline__ void solve_warp_body(const Params& P, int s, int pr, int lane, int64_t ld,
                                                const double* __restrict__ jac, const T* __restrict__ LU,
                                                const unsigned char* __restrict__ piv, const T* __restrict__ G,
                                                const double* x, const double* r0, const double* r1, double* o0,
                                                double* o1, T (*A)[PADL], int NP, int bsec) {
    constexpr bool INV = std::is_same<T, float>::value;
    int perm = lane, ipos = lane;
    const double* rr[2] = {r0, r1};
    double* oo[2] = {o0, o1};
    // b = dc/dtheta of the problem's design entry bsec
    const T bval = (T)(-P.u_max * M_PI * 0.5 * x[(int64_t)NSC * ld + (int64_t)bsec * NP + pr]);
    const bool row = lane < NV;
    T y[NRHS];
#pragma unroll
    for (int k = 0; k < NRHS; ++k) y[k] = T(0);
    typename std::conditional<INV, InvRowFetch, LUPrefetch>::type ipre, icur;
    ipre.fetch(LU, piv, s, 0, lane);
    double rnext[NRHS];
#pragma unroll
    for (int k = 0; k < NRHS; ++k) rnext[k] = (rr[k] && row) ? rr[k][(int64_t)lane * ld + s] : 0.0;
    CouplingFetch cnext;
    cnext.fetch<false>(1, ld, s, lane, jac);
    // forward: w_n = r_n - C_n y_{n-1},  y_n = At_n^-1 w_n
    for (int n = 0; n < N_STAGES; ++n) {
        if constexpr (INV) icur = ipre;
        else ipre.commit(A, perm, ipos, lane);
        const CouplingFetch cc = cnext;
        T w[NRHS];
#pragma unroll
        for (int k = 0; k < NRHS; ++k)
            w[k] = rr[k] ? (T)rnext[k] : ((lane == R_H && stage_sec(n, P.nsec) == bsec) ? bval : T(0));
        if (n + 1 < N_STAGES) {
            ipre.fetch(LU, piv, s, n + 1, lane);
#pragma unroll
            for (int k = 0; k < NRHS; ++k)
                rnext[k] = (rr[k] && row) ? rr[k][(int64_t)(NR * (n + 1) + lane) * ld + s] : 0.0;
            cnext.fetch<false>(n + 1, ld, s, lane, jac);
        }
        if (n > 0) {
            // products of C_n's entries (entry q on lane q) with y_{n-1}, then subtracted in
            // each row in entry order
            const T cv = (T)cc.cv;
#pragma unroll
            for (int k = 0; k < NRHS; ++k) {
                const T pq = cv * shfl(y[k], cc.src);
#pragma unroll
                for (int i = 0; i < NBLWV; ++i) {
                    const T pp = shfl(pq, (cc.q0 + i) & 31);
                    if (i < cc.nb) w[k] -= pp;
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < NRHS; ++k) {
            if constexpr (INV) y[k] = icur.apply(w[k]);
            else y[k] = lu_apply_warp(A, perm, lane, w[k]);
            if (row) oo[k][(int64_t)(NV * n + lane) * ld + s] = (double)y[k];
        }
        __syncwarp();
    }
    // backward: x_n = y_n - G_n x_{n+1}   (y currently holds x_9 = y_9); the forward
    // values y_n and G_n of the next stage down are fetched one stage ahead
    T gnext[NABV];
    T ynext[NRHS];
    auto fetch_back = [&](int n) {
        const T* Gn = G + g_off(s, n);
#pragma unroll
        for (int a = 0; a < NABV; ++a) gnext[a] = row ? Gn[lane * NABV + a] : T(0);
#pragma unroll
        for (int k = 0; k < NRHS; ++k) ynext[k] = row ? (T)oo[k][(int64_t)(NV * n + lane) * ld + s] : T(0);
    };
    fetch_back(N_STAGES - 2);
    for (int n = N_STAGES - 2; n >= 0; --n) {
        T gc[NABV], yc[NRHS];
#pragma unroll
        for (int a = 0; a < NABV; ++a) gc[a] = gnext[a];
#pragma unroll
        for (int k = 0; k < NRHS; ++k) yc[k] = ynext[k];
        if (n > 0) fetch_back(n - 1);
#pragma unroll
        for (int k = 0; k < NRHS; ++k) {
            T acc = yc[k];
#pragma unroll
            for (int a = 0; a < NABV; ++a) {
                const T xa = shfl(y[k], abv_var(a));
                if (row) acc -= gc[a] * xa;
            }
            y[k] = acc;
            if (row) oo[k][(int64_t)(NV * n + lane) * ld + s] = (double)acc;
        }
    }
}

template <class T, int NRHS, int WPB = WPB_S>
__global__ void __launch_bounds__(32 * WPB) solve_warp_kernel(const Params P, int S, int64_t ld, const BView b,
                                                                const double* __restrict__ jac,
                                                                const T* __restrict__ AI,
                                                                const unsigned char* __restrict__ piv,
                                                                const T* __restrict__ G, const double* x,
                                                                const double* r0, const double* r1, double* o0,
                                                                double* o1, int bsec = 0) {
    __shared__ T sL[std::is_same<T, float>::value ? 1 : WPB][NV][PADL];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = blockIdx.x * WPB + warp;
    const int pr = live_prob(b, s, S, PS_ACT);
    if (pr < 0) return;
    solve_warp_body<T, NRHS>(P, s, pr, lane, ld, jac, AI, piv, G, x, r0, r1, o0, o1,
                            sL[std::is_same<T, float>::value ? 0 : warp], b.NP, bsec);
}

// stage unknown j -> its index among the 11 stream-from-above unknowns (-1: none)
__host__ __device__ constexpr int abv_index(int j) { return j < 9 ? j : (j == LL ? 9 : (j == LT ? 10 : -1)); }

// J_s^T v = g, one warp per scenario; g in primal layout (no d), out in row layout.
// With the block LU J = L U (L: diagonal blocks At_n, sub-diagonal C_n; U: identity
// diagonal, super-diagonal G_n = At_n^-1 B_n), J^T = U^T L^T:
//   forward   w_0 = g_0,  w_{n+1} = g_{n+1} - G_n^T w_n   (into stage n+1's 11 unknowns
//             that stage n reads: products with the stored G blocks, no block solve)
//   backward  v_9 = At_9^-T w_9,  v_n = At_n^-T (w_n - C_{n+1}^T v_{n+1})
// one transposed block solve per stage.  T as solve_warp_body's.
template <class T>
__device__ __forceinline__ void solve_t_warp_body(int s, int lane, int64_t ld, const double* __restrict__ jac,
                                                  const T* __restrict__ LU, const unsigned char* __restrict__ piv,
                                                  const T* __restrict__ G, const double* __restrict__ g,
                                                  double* out, T (*A)[PADL]) {
    constexpr bool INV = std::is_same<T, float>::value;
    int perm = lane, ipos = lane;
    const bool row = lane < NV;
    const int my_abv = abv_index(lane);   // lane j takes the product of column abv_index(j)
    // forward sweep with the G blocks (fetched one stage ahead); w_n kept in out
    T w = row ? (T)g[(int64_t)lane * ld + s] : T(0);
    if (row) out[(int64_t)lane * ld + s] = (double)w;
    T gn[NV];
    auto fetch_g = [&](int n) {
        const T* Gn = G + g_off(s, n);
#pragma unroll
        for (int i = 0; i < NV; ++i) gn[i] = lane < NABV ? Gn[i * NABV + lane] : T(0);
    };
    fetch_g(0);
    for (int n = 1; n < N_STAGES; ++n) {
        T gc[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) gc[i] = gn[i];
        if (n + 1 < N_STAGES) fetch_g(n);
        const T gnext = row ? (T)g[(int64_t)(NV * n + lane) * ld + s] : T(0);
        // lane a < 11: (G_{n-1}^T w_{n-1})_a = sum_i G_{n-1}[i][a] w_{n-1,i}
        T acc = T(0);
#pragma unroll
        for (int i = 0; i < NV; ++i) acc += gc[i] * shfl(w, i);
        const T t = shfl(acc, my_abv >= 0 ? my_abv : 0);
        w = gnext - (my_abv >= 0 ? t : T(0));
        if (row) out[(int64_t)(NV * n + lane) * ld + s] = (double)w;
    }
    // backward sweep: one transposed block solve per stage
    typename std::conditional<INV, InvColFetch, LUPrefetch>::type ipre, icur;
    ipre.fetch(LU, piv, s, N_STAGES - 1, lane);
    double rnext = row ? out[(int64_t)(NV * (N_STAGES - 1) + lane) * ld + s] : 0.0;
    CouplingFetch cnext;
    cnext.fetch<true>(N_STAGES - 1, ld, s, lane, jac);
    T v = T(0);
    for (int n = N_STAGES - 1; n >= 0; --n) {
        if constexpr (INV) icur = ipre;
        else ipre.commit(A, perm, ipos, lane);
        T rhs = (T)rnext;
        const CouplingFetch cc = cnext;
        if (n > 0) {
            ipre.fetch(LU, piv, s, n - 1, lane);
            rnext = row ? out[(int64_t)(NV * (n - 1) + lane) * ld + s] : 0.0;
            cnext.fetch<true>(n, ld, s, lane, jac);
        }
        if (n + 1 < N_STAGES) {
            // C_{n+1}^T v_{n+1}: entry q's product (lane q) subtracted from the stage-n
            // unknown it multiplies, each unknown's entries in table order
            const T pq = (T)cc.cv * shfl(v, cc.src);
#pragma unroll
            for (int i = 0; i < NBLWC; ++i) {
                const T pp = shfl(pq, cc.qi[i]);
                if (i < cc.nb) rhs -= pp;
            }
        }
        __syncwarp();
        if constexpr (INV) v = icur.apply(rhs);
        else v = lu_apply_t_warp(A, ipos, lane, rhs);
        if (row) out[(int64_t)(NR * n + lane) * ld + s] = (double)v;
        __syncwarp();
    }
}

template <class T, int WPB = WPB_S>
__global__ void __launch_bounds__(32 * WPB) solve_t_warp_kernel(int S, int64_t ld, const BView b,
                                                                const double* __restrict__ jac,
                                                                const T* __restrict__ AI,
                                                                const unsigned char* __restrict__ piv,
                                                                const T* __restrict__ G,
                                                                const double* __restrict__ g, double* out) {
    __shared__ T sL[std::is_same<T, float>::value ? 1 : WPB][NV][PADL];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = blockIdx.x * WPB + warp;
    if (live_prob(b, s, S, PS_ACT) < 0) return;
    solve_t_warp_body<T>(s, lane, ld, jac, AI, piv, G, g, out, sL[std::is_same<T, float>::value ? 0 : warp]);
}

}  // namespace absorber
