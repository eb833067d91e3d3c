// kernels_ldl.cuh -- regularised symmetric indefinite factorization of the scenario
// blocks (included once, by absorber_lib.cu).
//
// The scenario block of the primal-dual matrix with both regularisations of Wachter &
// Biegler (2006, Eq. (13) and Section 3.1),
//     K_s = [ W_s + Sigma_s + dw I , J_s^T ; J_s , -dc I ],
// is ordered stage by stage, each stage's 22 unknowns followed by its 22 rows, so that
// it is block tridiagonal with 44 x 44 blocks: diagonal blocks K_nn and coupling blocks
// E_n = K_{n+1,n} (the rows of stage n+1 against the unknowns of stage n, J_{n+1,n}, and
// the unknowns of stage n+1 against the rows of stage n, J_{n,n+1}^T).  The block LDL^T
// recurrence in stage order
//     Dt_0 = K_00,   Dt_n = K_nn - E_{n-1} Dt_{n-1}^-1 E_{n-1}^T,
// factors every Dt_n by the Bunch-Kaufman partial pivoting rule (1 x 1 and 2 x 2
// pivots; Bunch & Kaufman 1977, alpha = (1 + sqrt 17) / 8); by
// Sylvester's law the inertia of K_s is the sum of the inertias of the pivot blocks.
// Each Dt_n is kept as its explicit inverse for the block solves, and factored and inverted
// together by symmetric sweeps (Goodnight 1979): a pivot p replaces W_ij by W_ij - W_ip W_pj / W_pp, its
// row and column by W_ip / W_pp and W_pp by -1 / W_pp (2 x 2 pivots alike), and after every index
// W = -Dt^-1.  On the indices not swept yet W is the Schur complement the Bunch-Kaufman rule looks at,
// so pivots are taken where they stand, without interchanges.  Only the lower triangle is stored and
// updated: 990 entries, one multiply-add each per pivot index -- 44 000 per block where a triangular
// factorization with a dense inverse took 150 000 --, shared out evenly over two warps.
// The coupling has 43 nonzeros, between 16 indices of each stage, so E Dt^-1 E^T is formed from
// them (about 1 400 multiply-adds against 130 000 dense).
// Unlike the block LU of J_s this needs no square nonsingular J_s: it is the
// factorization for dc > 0 (Algorithm IC's branch for a singular Jacobian) and for
// solves that must count the inertia of every scenario block.  Two warps per scenario, FP64, the
// block in shared memory.  The FP64 pipe and the pivots' dependent steps bound it: 500 scenarios 1.18 ms
// (13.9 with dense couplings and a triangular factorization on one warp), a solve 67 us.
#pragma once

#include "kernels.cuh"
#include "vec_kernels.cuh"
#include "kernels_cond.cuh"

namespace absorber {

constexpr int NB = NV + NR;                        // unknowns of a stage block of K_s
constexpr int LDL_BLOCK = NB * (NB + 1) / 2;       // entries of a packed lower triangle
constexpr int LDL_T = 64;                          // threads of a scenario
constexpr int LDL_PER = (LDL_BLOCK + LDL_T - 1) / LDL_T;
constexpr int NCPL = 16, NCPLE = 43;               // coupled indices of a stage, nonzeros of a coupling block

__device__ inline int64_t ldl_off(int s, int n) { return ((int64_t)s * N_STAGES + n) * LDL_BLOCK; }
__device__ __forceinline__ int tri(int i, int j) { return i >= j ? i * (i + 1) / 2 + j : j * (j + 1) / 2 + i; }

// The coupling block E_{n-1} = K_{n,n-1}: row a of 16 (stage n: unknowns x0..x8, L, T, rows 7, 8, 9, 10, E)
// against column c of 16 (stage n-1: rows 0..8, E, unknowns y0..y3, V, T); its nonzeros k in row
// order.  Rows of stage n on the unknowns of stage n-1 (its stream from below) and, transposed, rows
// of stage n-1 on the unknowns of stage n (their stream from above).
__device__ __forceinline__ int cpl_row(int a) {   // index in stage n's block
    return a < 9 ? a : (a == 9 ? LL : (a == 10 ? LT : NV + (a == 15 ? R_E : a - 4)));
}
__device__ __forceinline__ int cpl_col(int c) {   // index in stage n-1's block
    return c < 9 ? NV + c : (c == 9 ? NV + R_E : (c < 14 ? LY + c - 10 : (c == 14 ? LV : LT)));
}
__device__ __forceinline__ int cpl_ptr(int a) { return a < 10 ? 2 * a : (a == 10 ? 28 : (a < 16 ? 29 + 2 * (a - 11) : 43)); }
__device__ __forceinline__ int cpl_cidx(int k) {   // column of nonzero k
    if (k < 18) return (k & 1) ? 9 : k >> 1;
    if (k < 28) return k - 18;
    if (k == 28) return 9;
    if (k < 37) return ((k - 29) & 1) ? 14 : 10 + (k - 29) / 2;
    return 10 + k - 37;
}
// value of nonzero k of E_{n-1}
__device__ __forceinline__ double cpl_value(int k, int64_t ld, int s, int n, const double* __restrict__ jac) {
    int r, lv;
    const bool abv = k < 29;
    if (k < 18) r = (k & 1) ? R_E : k >> 1, lv = AX + (k >> 1);
    else if (k < 28) r = k < 27 ? k - 18 : R_E, lv = AL;
    else if (k == 28) r = R_E, lv = AT;
    else if (k < 37) r = 7 + (k - 29) / 2, lv = ((k - 29) & 1) ? BV : BY + (k - 29) / 2;
    else r = R_E, lv = BY + k - 37;
    const int m = abv ? n - 1 : n;
    return jac[(int64_t)(c_segJ[m] + c_slotJ[stage_type(m)][r][lv]) * ld + s];
}

__device__ __forceinline__ int cpl_arow(int k) {   // row of nonzero k
    return k < 18 ? k >> 1 : (k < 28 ? 9 : (k == 28 ? 10 : (k < 37 ? 11 + (k - 29) / 2 : 15)));
}
// a <- a - the products t (one per nonzero) of row a; of column c
__device__ __forceinline__ double cpl_row_sub(const double* t, int a, double v) {
    const int k1 = cpl_ptr(a + 1);
    for (int k = cpl_ptr(a); k < k1; ++k) v -= t[k];
    return v;
}
__device__ __forceinline__ double cpl_col_sub(const double* t, int c, double v) {
    if (c < 9) return v - t[2 * c] - t[18 + c];
    if (c == 9) {
#pragma unroll
        for (int q = 0; q < 9; ++q) v -= t[2 * q + 1];
        return v - t[27] - t[28];
    }
    if (c < 14) return v - t[29 + 2 * (c - 10)] - t[37 + c - 10];
    if (c == 14) return v - t[30] - t[32] - t[34] - t[36] - t[41];
    return v - t[42];
}

// 1 / a by cond_recip inside its range
__device__ __forceinline__ double ldl_recip(double a) {
    const double m = fabs(a);
    return m > 1e-290 && m < 1e290 ? cond_recip(a) : 1.0 / a;
}

// the diagonal block K_nn: [W_nn + Sigma_n + dw I, J_nn^T; J_nn, -dc I] (W omitted when
// use_w is false), packed
__device__ inline void ldl_assemble_diag(double* W, int64_t ld, int s, int n, const double* __restrict__ jac,
                                         const double* __restrict__ hes, const double* __restrict__ sig, bool use_w,
                                         double dw, double dc) {
    const int tid = threadIdx.x;
    for (int e = tid; e < LDL_BLOCK; e += LDL_T) W[e] = 0.0;
    __syncthreads();
    const int t = stage_type(n);
    if (use_w)
        for (int k = tid; k < NHS; k += LDL_T) {
            const Ent e = c_hes[k];
            W[tri(e.r, e.c)] = hes[(int64_t)(NHS * n + e.slot) * ld + s];
        }
    const int base = c_segJ[n];
    for (int k = tid; k < c_nown[t]; k += LDL_T) {
        const Ent e = c_own[t][k];
        W[tri(NV + e.r, e.c)] = jac[(int64_t)(base + e.slot) * ld + s];
    }
    __syncthreads();
    if (tid < NV) {
        W[tri(tid, tid)] += sig[(int64_t)(NV * n + tid) * ld + s] + dw;
        W[tri(NV + tid, NV + tid)] = -dc;
    }
}

// the largest |entry| of column k over the indices not in done and other than k, and its lowest
// index (every lane of the warp gets both; each warp of the block for itself)
__device__ __forceinline__ double ldl_colmax(const double* W, int k, unsigned long long done, int& row) {
    const int lane = threadIdx.x & 31, i1 = lane + 32;
    const bool c0 = !((done >> lane) & 1ull) && lane != k, c1 = i1 < NB && !((done >> i1) & 1ull) && i1 != k;
    const unsigned long long a0 = c0 ? mag_key(W[tri(lane, k)]) : 0ull, a1 = c1 ? mag_key(W[tri(i1, k)]) : 0ull;
    const unsigned long long m = warp_max_key(key_max(a0, a1));
    const unsigned b0 = __ballot_sync(0xffffffffu, c0 && a0 == m), b1 = __ballot_sync(0xffffffffu, c1 && a1 == m);
    row = b0 ? __ffs((int)b0) - 1 : (b1 ? 31 + __ffs((int)b1) : k);
    return key_double(m);
}

// factor K_s of every active scenario (dw = PS_DW, dc = PS_DC of its problem): the
// inverses of Dt_0 .. Dt_9 (packed) to Dinv_g, and per scenario (partials at stage 0, the other
// stages 0) [2] positive, [3] negative, [6] zero pivots of K_s, [5] 1 if any pivot is zero.
// Only exactly zero pivots count as zero (a zero column of the trailing block, or a
// singular 2 x 2 pivot): near-singular blocks are factored, as LAPACK's Bunch-Kaufman
// does, and their inertia read from the signs.  One scenario per block.
__global__ void __launch_bounds__(LDL_T) ldl_factor_kernel(int S, int64_t ld, const BView b,
                                                           const double* __restrict__ jac,
                                                           const double* __restrict__ hes,
                                                           const double* __restrict__ sig, bool use_w,
                                                           double* __restrict__ Dinv_g, double* __restrict__ part) {
    __shared__ double W[LDL_BLOCK];
    __shared__ double u[2][NB], v[2][NB];   // pivot columns, and those times the pivot's inverse
    __shared__ double X[NCPL][NCPL + 1];    // Dt^-1 E^T between the coupled indices
    __shared__ double E[NCPLE];
    __shared__ short ij[LDL_BLOCK];
    const int tid = threadIdx.x;
    const int s = blockIdx.x;
    const int p = live_prob(b, s, S, PS_ACT);
    if (p < 0) return;   // the whole block
    for (int i = tid; i < NB; i += LDL_T)
        for (int j = 0; j <= i; ++j) ij[tri(i, j)] = (short)(i << 8 | j);
    const double alpha = 0.64038820320220756872;   // (1 + sqrt(17)) / 8
    const double dw = b.ps ? psv(b, PS_DW, p) : 0.0;
    const double dc = b.ps ? psv(b, PS_DC, p) : 0.0;
    int npos = 0, nneg = 0, nzero = 0;
    for (int n = 0; n < N_STAGES; ++n) {
        // W = K_nn - E Dt_{n-1}^-1 E^T; the last stage's W is -Dt_{n-1}^-1
        if (n > 0) {
            if (tid < NCPLE) E[tid] = cpl_value(tid, ld, s, n, jac);
            __syncthreads();
            for (int e = tid; e < NCPL * NCPL; e += LDL_T) {
                const int i = e / NCPL, a = e % NCPL, ci = cpl_col(i);
                double acc = 0.0;
                for (int k = cpl_ptr(a); k < cpl_ptr(a + 1); ++k) acc = fma(W[tri(ci, cpl_col(cpl_cidx(k)))], E[k], acc);
                X[i][a] = acc;
            }
            __syncthreads();
        }
        ldl_assemble_diag(W, ld, s, n, jac, hes, sig, use_w, dw, dc);
        __syncthreads();
        if (n > 0) {
            for (int e = tid; e < NCPL * NCPL; e += LDL_T) {
                const int a = e / NCPL, c = e % NCPL;
                if (cpl_row(c) > cpl_row(a)) continue;
                double acc = 0.0;
                for (int k = cpl_ptr(a); k < cpl_ptr(a + 1); ++k) acc = fma(E[k], X[cpl_cidx(k)][c], acc);
                W[tri(cpl_row(a), cpl_row(c))] += acc;
            }
            __syncthreads();
        }
        // sweeps: both warps take the same pivot decisions from shared memory
        unsigned long long done = 0ull;
        const unsigned long long all = (1ull << NB) - 1ull;
        while (done != all) {
            const int k = __ffsll((long long)~done) - 1;   // the first index left
            int r, r2;
            const double lam = ldl_colmax(W, k, done, r);
            const double akk = fabs(W[tri(k, k)]);
            int kind = 1, pv = k;
            if (!(fmax(akk, lam) > 0.0)) {
                kind = 0;   // zero column (or NaN): a zero pivot
            } else if (akk < alpha * lam) {
                const double sg = ldl_colmax(W, r, done, r2);
                if (akk * sg >= alpha * lam * lam) kind = 1;
                else if (fabs(W[tri(r, r)]) >= alpha * sg) pv = r;
                else kind = 2;
            }
            if (kind == 0) {
                // eliminated with a zero inverse
                ++nzero;
                __syncthreads();
                if (tid < NB) W[tri(tid, k)] = 0.0;
                done |= 1ull << k;
                __syncthreads();
                continue;
            }
            if (kind == 1) {
                const double d = W[tri(pv, pv)];
                if (!(fabs(d) > 0.0)) ++nzero;
                else if (d > 0.0) ++npos;
                else ++nneg;
                const double di = ldl_recip(d);
                if (tid < NB) {
                    const double a = tid == pv ? 0.0 : W[tri(tid, pv)];
                    u[0][tid] = a;
                    v[0][tid] = a * di;
                }
                __syncthreads();
#pragma unroll
                for (int t = 0; t < LDL_PER; ++t) {
                    const int e = tid + LDL_T * t;
                    if (e < LDL_BLOCK) W[e] = fma(-u[0][ij[e] >> 8], v[0][ij[e] & 255], W[e]);
                }
                __syncthreads();
                if (tid < NB) W[tri(tid, pv)] = tid == pv ? -di : v[0][tid];
                done |= 1ull << pv;
            } else {
                const double a = W[tri(k, k)], o = W[tri(k, r)], c = W[tri(r, r)];
                const double det = a * c - o * o;   // < 0 for a Bunch-Kaufman 2 x 2 pivot
                if (det < 0.0) {
                    ++npos;
                    ++nneg;
                } else if (det > 0.0) {
                    if (a > 0.0) npos += 2;
                    else nneg += 2;
                } else {
                    ++nzero;
                    if (a + c > 0.0) ++npos;
                    else if (a + c < 0.0) ++nneg;
                    else ++nzero;
                }
                const double idet = ldl_recip(det);
                const double i11 = c * idet, i12 = -o * idet, i22 = a * idet;
                if (tid < NB) {
                    const bool in = tid == k || tid == r;
                    const double w0 = in ? 0.0 : W[tri(tid, k)], w1 = in ? 0.0 : W[tri(tid, r)];
                    u[0][tid] = w0;
                    u[1][tid] = w1;
                    v[0][tid] = w0 * i11 + w1 * i12;
                    v[1][tid] = w0 * i12 + w1 * i22;
                }
                __syncthreads();
#pragma unroll
                for (int t = 0; t < LDL_PER; ++t) {
                    const int e = tid + LDL_T * t;
                    if (e < LDL_BLOCK) {
                        const int i = ij[e] >> 8, j = ij[e] & 255;
                        W[e] = fma(-u[1][i], v[1][j], fma(-u[0][i], v[0][j], W[e]));
                    }
                }
                __syncthreads();
                if (tid < NB) {
                    W[tri(tid, k)] = tid == k ? -i11 : (tid == r ? -i12 : v[0][tid]);
                    if (tid != k) W[tri(tid, r)] = tid == r ? -i22 : v[1][tid];
                }
                done |= (1ull << k) | (1ull << r);
            }
            __syncthreads();
        }
        double* dst = Dinv_g + ldl_off(s, n);
        for (int e = tid; e < LDL_BLOCK; e += LDL_T) dst[e] = -W[e];
    }
    if (tid < N_STAGES) {
        const int64_t plane = (int64_t)N_STAGES * ld;
        const int64_t o = (int64_t)tid * ld + s;
        const bool z = tid == 0;
        part[2 * plane + o] = z ? (double)npos : 0.0;
        part[3 * plane + o] = z ? (double)nneg : 0.0;
        part[5 * plane + o] = z ? (nzero > 0 ? 1.0 : 0.0) : 0.0;
        part[6 * plane + o] = z ? (double)nzero : 0.0;
    }
}

// v = K_s^-1 r of every active scenario with the inverses of ldl_factor_kernel:
// forward g_0 = r_0, g_n = r_n - E_{n-1} Dinv_{n-1} g_{n-1} (the 16 coupled entries only); backward
// x_9 = Dinv_9 g_9, x_n = Dinv_n (g_n - E_n^T x_{n+1}).  r: z part rz (primal layout), row part rc (row
// layout); rhs_b: r = [0; b] instead, b = dc/dd (the d entries of the hydraulic rows).
// Out: xz (primal layout, d slots untouched), xl (row layout); partial plane `pl` of each
// scenario: sgn * b^T x_l at stage 0 (the other stages 0).  fac_planes (the factorization's
// u = K_s^-1 [0; b], pl = 0): plane 1 zero and plane 4 the scenario's d-d Hessian entry
// (hes, or 0 without), as the block-LU path's Schur sums lay them out; otherwise (a solve,
// pl = 2) planes 0, 1 and 3 zero.  One scenario per block; the next stage's inverse is on its way to
// registers while a stage is worked on.
__global__ void __launch_bounds__(LDL_T) ldl_solve_kernel(int S, int64_t ld, const BView b,
                                                          const double* __restrict__ jac,
                                                          const double* __restrict__ Dinv_g,
                                                          const double* __restrict__ rz, const double* __restrict__ rc,
                                                          bool rhs_b, double* __restrict__ xz, double* __restrict__ xl,
                                                          double* __restrict__ part, int pl, double sgn, bool fac_planes,
                                                          const double* __restrict__ hes) {
    __shared__ double D[LDL_BLOCK];
    __shared__ double G[N_STAGES][NB], H[NB];
    __shared__ double E[N_STAGES][NCPLE];   // E[n]: the coupling of stages n and n - 1
    __shared__ double T[NCPLE];             // products of a coupling's nonzeros
    __shared__ double sb[2];
    const int tid = threadIdx.x;
    // the thread's nonzero (its column; its row's index) and its coupled row's and column's indices
    const int cidx = tid < NCPLE ? cpl_cidx(tid) : 0, krow = tid < NCPLE ? cpl_row(cpl_arow(tid)) : 0;
    const int arow = cpl_row(tid & 15), acol = cpl_col(tid & 15);
    const int s = blockIdx.x;
    const int p = live_prob(b, s, S, PS_ACT);
    if (p < 0) return;   // the whole block
    double nx[LDL_PER];
    auto fetch = [&](int n) {
        const double* src = Dinv_g + ldl_off(s, n);
#pragma unroll
        for (int t = 0; t < LDL_PER; ++t) nx[t] = tid + LDL_T * t < LDL_BLOCK ? src[tid + LDL_T * t] : 0.0;
    };
    auto commit = [&]() {
#pragma unroll
        for (int t = 0; t < LDL_PER; ++t)
            if (tid + LDL_T * t < LDL_BLOCK) D[tid + LDL_T * t] = nx[t];
    };
    fetch(0);
    for (int e = tid; e < N_STAGES * NB; e += LDL_T) {
        const int n = e / NB, i = e - n * NB;
        double v;
        if (rhs_b) v = (i == NV + R_H) ? jac[(int64_t)(c_segJ[n] + c_dslot[stage_type(n)]) * ld + s] : 0.0;
        else v = i < NV ? rz[(int64_t)(NV * n + i) * ld + s] : rc[(int64_t)(NR * n + i - NV) * ld + s];
        G[n][i] = v;
    }
    for (int e = tid; e < (N_STAGES - 1) * NCPLE; e += LDL_T)
        E[1 + e / NCPLE][e % NCPLE] = cpl_value(e % NCPLE, ld, s, 1 + e / NCPLE, jac);
    // forward: four threads per coupled row of the inverse
    for (int n = 1; n < N_STAGES; ++n) {
        commit();
        __syncthreads();
        fetch(n);   // the next stage's (the last: the backward sweep's first)
        const int c = tid >> 2, ci = cpl_col(c);
        double acc = 0.0;
#pragma unroll
        for (int j = 0; j < NB / 4; ++j) acc = fma(D[tri(ci, 4 * j + (tid & 3))], G[n - 1][4 * j + (tid & 3)], acc);
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if ((tid & 3) == 0) H[c] = acc;
        __syncthreads();
        if (tid < NCPLE) T[tid] = E[n][tid] * H[cidx];
        __syncthreads();
        if (tid < NCPL) G[n][arow] = cpl_row_sub(T, tid, G[n][arow]);
        __syncthreads();
    }
    // backward
    for (int n = N_STAGES - 1; n >= 0; --n) {
        commit();
        if (tid < NB) H[tid] = G[n][tid];
        __syncthreads();
        if (n > 0) fetch(n - 1);
        if (n + 1 < N_STAGES) {
            if (tid < NCPLE) T[tid] = E[n + 1][tid] * G[n + 1][krow];
            __syncthreads();
            if (tid < NCPL) H[acol] = cpl_col_sub(T, tid, H[acol]);
            __syncthreads();
        }
        if (tid < NB) {
            double a0 = 0.0, a1 = 0.0;
#pragma unroll
            for (int j = 0; j < NB; j += 2) {
                a0 = fma(D[tri(tid, j)], H[j], a0);
                a1 = fma(D[tri(tid, j + 1)], H[j + 1], a1);
            }
            G[n][tid] = a0 + a1;
        }
        __syncthreads();
    }
    double bs = 0.0;
    for (int e = tid; e < N_STAGES * NB; e += LDL_T) {
        const int n = e / NB, i = e - n * NB;
        if (i < NV) xz[(int64_t)(NV * n + i) * ld + s] = G[n][i];
        else xl[(int64_t)(NR * n + i - NV) * ld + s] = G[n][i];
        if (i == NV + R_H) bs += jac[(int64_t)(c_segJ[n] + c_dslot[stage_type(n)]) * ld + s] * G[n][i];
    }
    // the threads' terms combined in a fixed order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) bs += __shfl_xor_sync(0xffffffffu, bs, o);
    if ((tid & 31) == 0) sb[tid >> 5] = bs;
    __syncthreads();
    if (tid < N_STAGES) {
        const int64_t plane = (int64_t)N_STAGES * ld;
        const int64_t o = (int64_t)tid * ld + s;
        part[pl * plane + o] = tid == 0 ? sgn * (sb[0] + sb[1]) : 0.0;
        if (fac_planes) {
            part[1 * plane + o] = 0.0;
            part[4 * plane + o] = (tid == 0 && hes) ? hes[(int64_t)(NHS * N_STAGES) * ld + s] : 0.0;
        } else {
            part[0 * plane + o] = 0.0;
            part[1 * plane + o] = 0.0;
            part[3 * plane + o] = 0.0;
        }
    }
}

// the back-substitution of the Schur step on d: x = v - u dd for the z part (dz, d slots
// untouched) and the row part (dl), dd the problem's (dz's d slot).  One thread per
// (scenario, stage).
__global__ void __launch_bounds__(128) ldl_back_kernel(int S, int64_t ld, const BView b, const double* __restrict__ uz,
                                                       const double* __restrict__ ul, double* __restrict__ dz,
                                                       double* __restrict__ dl) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = blockIdx.y;
    const int p = live_prob(b, s, S, PS_ACT);
    if (p < 0) return;
    const double dd = dz[(int64_t)NSC * ld + p];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const int64_t oz = (int64_t)(NV * n + j) * ld + s, ol = (int64_t)(NR * n + j) * ld + s;
        dz[oz] = fma(-uz[oz], dd, dz[oz]);
        dl[ol] = fma(-ul[ol], dd, dl[ol]);
    }
}

// (H v)_j's terms of unknown j (H = the stage's Hessian block), subtracted from a
template <int j>
__device__ __forceinline__ double hv_col(int64_t ld, const double* __restrict__ h, const double* __restrict__ vn,
                                         double a) {
    static_for<0, NV>([&](auto I) {
        constexpr int i = decltype(I)::value, hi = i > j ? i : j, lo = i > j ? j : i;
        if constexpr (hes_has(hi, lo)) a = fma(-h[(int64_t)c_slotH[hi][lo] * ld], vn[(int64_t)i * ld], a);
    });
    return a;
}

// the KKT residual of the regularised system, every term formed directly:
// rho_z = r_z - (W + Sigma + dw I) dz - J^T dl,  rho_c = r_c - J dz - b dd + dc dl;
// partials as kkt_residual_kernel's: [0] max|rho_z|, [1] max|rho_c|, [2] the stage's
// hydraulic dl, [3] max|r_z|, [4] max|r_c|.  cz (optional): a correction whose design entry is not in
// dz yet.  Warp = group of rows and unknowns, lane = scenario.
template <int G>
__device__ __forceinline__ void residual_reg_group(int64_t ld, const StageJac& J, const double* __restrict__ hes,
                                                   const double* __restrict__ sig, bool use_w, double dw, double dc,
                                                   const double* __restrict__ dz, const double* __restrict__ dl,
                                                   double dd, const double* __restrict__ rz,
                                                   const double* __restrict__ rc, double* __restrict__ rhoz,
                                                   double* __restrict__ rhoc, int s, int n, double (&v)[5]) {
    unsigned long long k0 = 0, k1 = 0, k3 = 0, k4 = 0;
    static_for<0, NV>([&](auto C) {
        constexpr int j = decltype(C)::value;
        if constexpr (col_grp(j) == G) {
            const int64_t o = (int64_t)(NV * n + j) * ld + s;
            const double r0 = rz[o];
            double a = fma(-(sig[o] + dw), dz[o], r0);
            if (use_w) a = hv_col<j>(ld, hes + (int64_t)(NHS * n) * ld + s, dz + (int64_t)(NV * n) * ld + s, a);
            a = jt_col<-1, j>(J, dl, s, n, a);
            rhoz[o] = a;
            k0 = key_max(k0, mag_key(a));
            k3 = key_max(k3, mag_key(r0));
        }
    });
    static_for<0, NR>([&](auto R) {
        constexpr int r = decltype(R)::value;
        if constexpr (row_grp(r) == G) {
            const int64_t o = (int64_t)(NR * n + r) * ld + s;
            const double r0 = rc[o];
            const double c = jv_row<r>(J, dz, dd, s, n, fma(dc, dl[o], r0));
            rhoc[o] = c;
            k1 = key_max(k1, mag_key(c));
            k4 = key_max(k4, mag_key(r0));
        }
    });
    if (k1 > 0x7ff0000000000000ull) k0 = k1;   // NaN
    v[0] = key_double(k0);
    v[1] = key_double(k1);
    v[3] = key_double(k3);
    v[4] = key_double(k4);
}

__global__ void __launch_bounds__(128) kkt_residual_reg_kernel(int S, int64_t ld, const BView b,
                                                               const double* __restrict__ jac,
                                                               const double* __restrict__ hes,
                                                               const double* __restrict__ sig, bool use_w,
                                                               const double* __restrict__ dz,
                                                               const double* __restrict__ dl,
                                                               const double* __restrict__ cz,
                                                               const double* __restrict__ rz,
                                                               const double* __restrict__ rc, double* __restrict__ rhoz,
                                                               double* __restrict__ rhoc, double* part) {
    __shared__ double sm[QS][5][32];
    const int gq = threadIdx.x >> 5;
    const int s = blockIdx.x * QS_SCEN + (threadIdx.x & 31);
    const int n = blockIdx.y;
    const int p = live_prob(b, s, S, PS_ACT);
    const bool live = p >= 0;
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (live) {
        const double dw = b.ps ? psv(b, PS_DW, p) : 0.0;
        const double dc = b.ps ? psv(b, PS_DC, p) : 0.0;
        const double dd = dz[(int64_t)NSC * ld + p] + (cz ? cz[(int64_t)NSC * ld + p] : 0.0);
        const StageJac J(jac, ld, s, n);
#define RG(g) residual_reg_group<g>(ld, J, hes, sig, use_w, dw, dc, dz, dl, dd, rz, rc, rhoz, rhoc, s, n, v)
        switch (gq) {
            case 0: RG(0); break;
            case 1: RG(1); break;
            case 2: RG(2); break;
            default: RG(3); break;
        }
#undef RG
    }
    constexpr int ops[5] = {RMAX, RMAX, RSUM, RMAX, RMAX};   // [2] is set below
    group_combine<5, 5>(v, sm, ops);
    if (!live || gq != 0) return;
    v[2] = dl[(int64_t)(NR * n + R_H) * ld + s];
    store_partials<5>(v, part, ld, s, n);
}

}  // namespace absorber
