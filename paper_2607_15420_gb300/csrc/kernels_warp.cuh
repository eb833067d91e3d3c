// kernels_warp.cuh -- warp-cooperative block solves with stage-block inverses: the solves of
// the tensor-core FP32 factor (factor_gj_tc_kernel, kernels_tc.cuh), and what that kernel's
// assembly shares with them.
//
// One warp per scenario; vectors live one entry per lane, broadcasts are warp shuffles.
// Factor storage is per scenario and contiguous (internal layout, not part of the C ABI): the
// inverse [s][n][22][22], G[s][n][22][11] and the row order piv[s][n][22][2] (see PIV_BYTES),
// so every warp access to the factors is coalesced.
#pragma once

#include "kernels.cuh"

namespace absorber {

constexpr int NCA = NV + NABV;    // augmented columns [A_n | B_n]
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
// LU holds the stage-block inverses: each block solve is a matrix-vector product.  The block
// solves of scenario s (problem pr) by its warp.
template <int NRHS>
__device__ __forceinline__ void solve_warp_body(const Params& P, int s, int pr, int lane, int64_t ld,
                                                const double* __restrict__ jac, const float* __restrict__ LU,
                                                const unsigned char* __restrict__ piv, const float* __restrict__ G,
                                                const double* x, const double* r0, const double* r1, double* o0,
                                                double* o1, int NP, int bsec) {
    using T = float;
    const double* rr[2] = {r0, r1};
    double* oo[2] = {o0, o1};
    // b = dc/dtheta of the problem's design entry bsec
    const T bval = (T)(-P.u_max * M_PI * 0.5 * x[(int64_t)NSC * ld + (int64_t)bsec * NP + pr]);
    const bool row = lane < NV;
    T y[NRHS];
#pragma unroll
    for (int k = 0; k < NRHS; ++k) y[k] = T(0);
    InvRowFetch ipre;
    ipre.fetch(LU, piv, s, 0, lane);
    double rnext[NRHS];
#pragma unroll
    for (int k = 0; k < NRHS; ++k) rnext[k] = (rr[k] && row) ? rr[k][(int64_t)lane * ld + s] : 0.0;
    CouplingFetch cnext;
    cnext.fetch<false>(1, ld, s, lane, jac);
    // forward: w_n = r_n - C_n y_{n-1},  y_n = At_n^-1 w_n
    for (int n = 0; n < N_STAGES; ++n) {
        const InvRowFetch icur = ipre;
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
            y[k] = icur.apply(w[k]);
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

template <int NRHS, int WPB = WPB_S>
__global__ void __launch_bounds__(32 * WPB) solve_warp_kernel(const Params P, int S, int64_t ld, const BView b,
                                                                const double* __restrict__ jac,
                                                                const float* __restrict__ AI,
                                                                const unsigned char* __restrict__ piv,
                                                                const float* __restrict__ G, const double* x,
                                                                const double* r0, const double* r1, double* o0,
                                                                double* o1, int bsec = 0) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = blockIdx.x * WPB + warp;
    const int pr = live_prob(b, s, S, PS_ACT);
    if (pr < 0) return;
    solve_warp_body<NRHS>(P, s, pr, lane, ld, jac, AI, piv, G, x, r0, r1, o0, o1, b.NP, bsec);
}

// stage unknown j -> its index among the 11 stream-from-above unknowns (-1: none)
__host__ __device__ constexpr int abv_index(int j) { return j < 9 ? j : (j == LL ? 9 : (j == LT ? 10 : -1)); }

// J_s^T v = g, one warp per scenario; g in primal layout (no d), out in row layout.
// With the block LU J = L U (L: diagonal blocks At_n, sub-diagonal C_n; U: identity
// diagonal, super-diagonal G_n = At_n^-1 B_n), J^T = U^T L^T:
//   forward   w_0 = g_0,  w_{n+1} = g_{n+1} - G_n^T w_n   (into stage n+1's 11 unknowns
//             that stage n reads: products with the stored G blocks, no block solve)
//   backward  v_9 = At_9^-T w_9,  v_n = At_n^-T (w_n - C_{n+1}^T v_{n+1})
// one transposed block solve per stage.
__device__ __forceinline__ void solve_t_warp_body(int s, int lane, int64_t ld, const double* __restrict__ jac,
                                                  const float* __restrict__ LU, const unsigned char* __restrict__ piv,
                                                  const float* __restrict__ G, const double* __restrict__ g,
                                                  double* out) {
    using T = float;
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
    InvColFetch ipre;
    ipre.fetch(LU, piv, s, N_STAGES - 1, lane);
    double rnext = row ? out[(int64_t)(NV * (N_STAGES - 1) + lane) * ld + s] : 0.0;
    CouplingFetch cnext;
    cnext.fetch<true>(N_STAGES - 1, ld, s, lane, jac);
    T v = T(0);
    for (int n = N_STAGES - 1; n >= 0; --n) {
        const InvColFetch icur = ipre;
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
        v = icur.apply(rhs);
        if (row) out[(int64_t)(NR * n + lane) * ld + s] = (double)v;
        __syncwarp();
    }
}

template <int WPB = WPB_S>
__global__ void __launch_bounds__(32 * WPB) solve_t_warp_kernel(int S, int64_t ld, const BView b,
                                                                const double* __restrict__ jac,
                                                                const float* __restrict__ AI,
                                                                const unsigned char* __restrict__ piv,
                                                                const float* __restrict__ G,
                                                                const double* __restrict__ g, double* out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = blockIdx.x * WPB + warp;
    if (live_prob(b, s, S, PS_ACT) < 0) return;
    solve_t_warp_body(s, lane, ld, jac, AI, piv, G, g, out);
}

}  // namespace absorber
