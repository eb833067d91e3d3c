// mlp_lib.cu -- the warm-start network of the learned warm start: a 3 -> 256 -> 256 ->
// 256 -> 440 perceptron with GELU activations, bfloat16 weights and FP32 accumulation,
// trained on the GPU by the kernels below (forward, reverse-mode backward, Adam).
//
//   a0 = (X - in_shift) / in_scale
//   a_l = gelu(a_{l-1} W_l^T + b_l),  l = 1..3;   gelu(x) = x Phi(x) (exact erf form)
//   yhat = a3 W4^T + b4                 (normalised outputs; raw = yhat * out_scale + out_shift)
//   loss = sum (yhat - (Y - out_shift) / out_scale)^2 / (2 n 440)
// The weight matrices enter every product as bfloat16 copies (round to nearest even)
// of FP32 master weights; biases, activations and sums are FP32.  Gradients are taken
// with respect to the rounded weights and applied to the masters by Adam (Kingma & Ba
// 2015, Algorithm 1).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "absorber.h"
#include "kernels_umma.cuh"

namespace {

constexpr int NIN = ABS_MLP_IN, NH = ABS_MLP_HIDDEN, NOUT = ABS_MLP_OUT;
constexpr int64_t NPAR = ABS_MLP_PARAMS;
// layer l: fan-in, fan-out, offsets of W_l ([out][in], row-major) and b_l in the flat vector
__host__ __device__ constexpr int l_in(int l) { return l == 0 ? NIN : NH; }
__host__ __device__ constexpr int l_out(int l) { return l == 3 ? NOUT : NH; }
__host__ __device__ constexpr int64_t off_w(int l) { return l == 0 ? 0 : off_w(l - 1) + l_in(l - 1) * l_out(l - 1) + l_out(l - 1); }
__host__ __device__ constexpr int64_t off_b(int l) { return off_w(l) + l_in(l) * l_out(l); }
static_assert(off_b(3) + NOUT == NPAR, "parameter layout");
static_assert(off_w(1) % 4 == 0 && off_w(2) % 4 == 0 && off_w(3) % 4 == 0 && NH % 4 == 0 && NOUT % 4 == 0,
              "four consecutive weights of layers 2-4 are read and written together");

constexpr int CHUNK_ROWS = 8192;   // inference rows per pass (bounds the activation workspace)

thread_local std::string g_mlp_err = "no error";

}  // namespace

struct abs_mlp {
    int dev = 0;
    float* theta = nullptr;          // FP32 master parameters [NPAR]
    __nv_bfloat16* wb = nullptr;     // bfloat16 copies at the same offsets (weights only are read)
    __nv_bfloat16* wt = nullptr;     // W2..W4's again as 128 x 128 chunks in the tensor cores' layout
    float* grad = nullptr;           // [NPAR]
    float* m = nullptr;              // Adam moments [NPAR]
    float* v = nullptr;
    int64_t step = 0;                // Adam steps taken
    float* norm = nullptr;           // device: in_shift[3], in_scale[3], out_shift[440], out_scale[440]
    double hnorm[2 * NIN + 2 * NOUT];
    // activation workspace for cap rows
    int64_t cap = 0;
    float* a0 = nullptr;             // [cap][3] normalised inputs
    float* z[3] = {nullptr, nullptr, nullptr};   // pre-activations [cap][256]
    float* a[3] = {nullptr, nullptr, nullptr};   // activations [cap][256]
    float* yh = nullptr;             // [cap][440]
    float* g = nullptr;              // dloss/dyhat [cap][440]
    float* da = nullptr;             // [cap][256]
    float* dz = nullptr;             // [cap][256]
    float* xb = nullptr;             // gathered minibatch inputs [cap][3]
    float* ybt = nullptr;            // gathered minibatch targets [cap][440]
    int* perm = nullptr;             // [perm_cap]
    int64_t perm_cap = 0;
    double* lpart = nullptr;         // loss partial sums
    int64_t lpart_cap = 0;
    double* lacc = nullptr;          // per-epoch loss accumulators
    int64_t lacc_cap = 0;
    bool tc = true;                  // tensor-core products for the 256-input layers
    int* hfault = nullptr;           // mapped host flag: a tensor-core wait gave up
    int* dfault = nullptr;
    std::string err = "no error";
};

namespace {

abs_status mfail(abs_mlp* n, abs_status st, const std::string& msg) {
    if (n) n->err = msg;
    g_mlp_err = msg;
    return st;
}

#define MCK(call)                                                                         \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess)                                                            \
            return mfail(net, e_ == cudaErrorMemoryAllocation ? ABS_ERR_OOM : ABS_ERR_CUDA, \
                         std::string(#call) + ": " + cudaGetErrorString(e_));             \
    } while (0)

abs_status mlaunch(abs_mlp* net) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return mfail(net, ABS_ERR_CUDA, std::string("kernel launch: ") + cudaGetErrorString(e));
    return ABS_OK;
}

__device__ __forceinline__ float gelu_f(float x) { return x * 0.5f * (1.0f + erff(x * 0.70710678118654752f)); }

__device__ __forceinline__ float gelu_prime_f(float x) {
    return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// the chunks of W2, W3 (two groups of 128 outputs each) and W4 (four groups, the outputs past the
// 440th zero), each group in two halves of its inputs
constexpr int NGROUP = 2 + 2 + 4, NCHUNK = 2 * NGROUP;
constexpr int CHUNK_ELS = umma::TILE_BYTES / 2;
// element (output o, input k) of layer l = 1, 2, 3 in wt
__device__ __forceinline__ int tile_element(int l, int o, int k) {
    const int g = (l - 1) * 2 + o / umma::TO;
    return (2 * g + k / umma::KC) * CHUNK_ELS + (int)(umma::w_off(o % umma::TO, k % umma::KC) >> 1);
}
// where weight i of the flat parameters lies in wt (-1: W1 or a bias)
__device__ __forceinline__ int tile_index(int64_t i) {
#pragma unroll
    for (int l = 1; l < 4; ++l) {
        const int64_t e = i - off_w(l);
        if (e >= 0 && e < (int64_t)l_out(l) * NH) return tile_element(l, (int)(e / NH), (int)(e % NH));
    }
    return -1;
}

enum { EPI_BIAS_GELU = 1, EPI_BIAS = 2, EPI_DENORM = 4 };

constexpr int BM = 64, BN = 64, BK = 16, GT = 256;

// C[m][n] = sum_k A[m][k] W[n][k] on the CUDA cores (the first layer, and every layer with the tensor
// cores switched off): A FP32 [M][K], W bfloat16 [N][K]; 64x64 tile per block, 4x4 outputs per
// thread, K in steps of 16 staged in shared memory.  Epilogues:
//   EPI_BIAS_GELU  Z = acc + bias[n] (stored), C = gelu(Z)
//   EPI_BIAS       C = acc + bias[n]
//   EPI_DENORM     C = (acc + bias[n]) * scale[n] + shift[n]
// Row-major C and Z with leading dimension N.
template <int EPI>
__global__ void __launch_bounds__(GT) gemm_kernel(int M, int N, int K, const float* __restrict__ A,
                                                  const __nv_bfloat16* __restrict__ W,
                                                  const float* __restrict__ bias, float* __restrict__ Z,
                                                  float* __restrict__ C, const float* __restrict__ scale,
                                                  const float* __restrict__ shift) {
    __shared__ __align__(16) float As[BK][BM + 4];
    __shared__ __align__(16) float Bs[BK][BN + 4];
    const int tid = threadIdx.x;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int tr = tid / 16, tc = tid % 16;   // this thread's 4 rows tr*4.. and 4 columns tc*4..
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
    for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
        for (int r = 0; r < (BM * BK) / GT; ++r) {
            const int e = tid + r * GT, mm = e / BK, kk = e % BK;
            const int gm = m0 + mm, gk = k0 + kk;
            As[kk][mm] = (gm < M && gk < K) ? A[(int64_t)gm * K + gk] : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < (BN * BK) / GT; ++r) {
            const int e = tid + r * GT, nn = e / BK, kk = e % BK;
            const int gn = n0 + nn, gk = k0 + kk;
            Bs[kk][nn] = (gn < N && gk < K) ? __bfloat162float(W[(int64_t)gn * K + gk]) : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            const float4 av = *reinterpret_cast<const float4*>(&As[kk][tr * 4]);
            const float4 bv = *reinterpret_cast<const float4*>(&Bs[kk][tc * 4]);
            const float ar[4] = {av.x, av.y, av.z, av.w};
            const float br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ar[i], br[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int gm = m0 + tr * 4 + i;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int gn = n0 + tc * 4 + j;
            if (gn >= N) continue;
            const int64_t o = (int64_t)gm * N + gn;
            float vv = acc[i][j] + bias[gn];
            if (EPI == EPI_BIAS_GELU) {
                Z[o] = vv;
                vv = gelu_f(vv);
            } else if (EPI == EPI_DENORM) {
                vv = vv * scale[gn] + shift[gn];
            }
            C[o] = vv;
        }
    }
}

template <int EPI>
abs_status gemm(abs_mlp* net, cudaStream_t st, int M, int N, int K, const float* A, const __nv_bfloat16* W, float* C,
                const float* bias, float* Z = nullptr, const float* scale = nullptr, const float* shift = nullptr) {
    if (M <= 0 || N <= 0) return ABS_OK;
    const dim3 grid((unsigned)((N + BN - 1) / BN), (unsigned)((M + BM - 1) / BM));
    gemm_kernel<EPI><<<grid, GT, 0, st>>>(M, N, K, A, W, bias, Z, C, scale, shift);
    return mlaunch(net);
}

// The whole forward pass of 64 samples per block, the products of layers 2-4 on the tensor cores
// (kernels_umma.cuh).  The activations stay on chip: their three bfloat16 terms in shared memory
// (96 KB), the weights streaming past them in 16 chunks of 128 outputs x 128 inputs (32 KB each, bulk
// copies of the tiled weights wt into a ring of three), the accumulators in two tensor-memory buffers of
// 192 columns, one per group of 128 outputs.  Warps 0-15: the layers' biases and GELU and the split into
// terms, 32 outputs x 16 samples of every group each, while the next group's MMAs run; a layer's
// activations are kept in registers until its last MMA has read the previous ones.  Warp 16: one
// thread loads the chunks and issues the 8 MMAs of each.  Biases, scales and W1
// wait in shared memory.
// One block's chain of 16 chunks bounds it, not the MMAs' rate or memory: 26 us for 1 to 9728 samples
// (one wave of 152 blocks), 5000 of them 94 us as a launch per layer.
// Every wait is bounded (wait_limit polls); when one gives up the block sets fault and leaves, its
// outputs unwritten.  idle (the self-test of that path): no MMA is issued.
// TRAIN: also a0, the pre-activations z and activations a of the layers, and normalised outputs;
// otherwise outputs de-normalised.
constexpr int FWD_E = 512, FWD_T = FWD_E + 32;
// constants in shared memory (floats): biases of layers 1-4, output shift and scale, W1, the block's
// normalised inputs
constexpr int FC_B = 0, FC_OUT = 3 * NH + NOUT, FC_W1 = FC_OUT + 2 * NOUT, FC_X = FC_W1 + NIN * NH,
              FC_COUNT = FC_X + NIN * umma::TR;
constexpr int FWD_SMEM = umma::ACT_BYTES + 3 * umma::TILE_BYTES + 4 * FC_COUNT + 1024;
static_assert(FWD_SMEM <= 227 * 1024, "shared memory of a block");
struct FwdTrain {
    float *a0, *z[3], *a[3];
};
template <bool TRAIN>
__global__ void __launch_bounds__(FWD_T, 1) network_forward_kernel(int M, const float* __restrict__ X,
                                                                   const float* __restrict__ norm,
                                                                   const float* __restrict__ theta,
                                                                   const __nv_bfloat16* __restrict__ wb,
                                                                   const __nv_bfloat16* __restrict__ wt,
                                                                   float* __restrict__ Y, const FwdTrain tr,
                                                                   int* __restrict__ fault, int idle,
                                                                   long long wait_limit) {
    using namespace umma;
    extern __shared__ unsigned char tc_smem[];
    __shared__ __align__(8) uint64_t bars[3 + 3 + 2 + 2 + 1];
    __shared__ uint32_t tbase;
    unsigned char* sm = (unsigned char*)(((uintptr_t)tc_smem + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * TR;
    const uint32_t sx = smem_u32(sm), sw = sx + ACT_BYTES;
    const uint32_t wfull = smem_u32(&bars[0]), wfree = smem_u32(&bars[3]), mdone = smem_u32(&bars[6]),
                   tfree = smem_u32(&bars[8]), aready = smem_u32(&bars[10]);
    if (warp == 0) {
        tmem_alloc(smem_u32(&tbase), TMEM_COLS);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < 3; ++i) {
            mbar_init(wfull + 8 * i, 1);
            mbar_init(wfree + 8 * i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(mdone + 8 * i, 1);
            mbar_init(tfree + 8 * i, FWD_E);
        }
        mbar_init(aready, FWD_E);
    }
    float* fc = reinterpret_cast<float*>(sm + ACT_BYTES + 3 * TILE_BYTES);
    for (int i = tid; i < FC_COUNT; i += FWD_T) {
        float f;
        if (i < FC_OUT) {
            f = theta[i < 3 * NH ? (i < NH ? off_b(0) + i : (i < 2 * NH ? off_b(1) + i - NH : off_b(2) + i - 2 * NH))
                                 : off_b(3) + i - 3 * NH];
        } else if (i < FC_W1) {
            f = norm[2 * NIN + i - FC_OUT];
        } else if (i < FC_X) {
            f = __bfloat162float(wb[off_w(0) + i - FC_W1]);
        } else {
            const int e = i - FC_X, r = e / NIN, k = e % NIN;
            f = 0.0f;
            if (m0 + r < M) {
                f = (X[(int64_t)(m0 + r) * NIN + k] - norm[k]) / norm[NIN + k];
                if (TRAIN) tr.a0[(int64_t)(m0 + r) * NIN + k] = f;
            }
        }
        fc[i] = f;
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = tbase;
    bool ok = true;
    if (warp == FWD_E / 32) {
        if (lane == 0) {
            int loaded = 0, taken = 0;   // chunks asked for / arrived
            const uint64_t dx = desc(sx, X_LBO, SBO), dw = desc(sw, W_LBO, SBO);
            const uint32_t xlo = (uint32_t)dx, xhi = (uint32_t)(dx >> 32), wlo = (uint32_t)dw, whi = (uint32_t)(dw >> 32);
            auto load = [&]() {
                const uint32_t bar = wfull + 8 * (loaded % 3);
                mbar_expect(bar, TILE_BYTES);
                bulk_load(sw + (loaded % 3) * TILE_BYTES, wt + (int64_t)loaded * CHUNK_ELS, TILE_BYTES, bar);
                ++loaded;
            };
            for (int i = 0; i < 3; ++i) load();
            for (int g = 0; g < NGROUP && ok; ++g) {
                // a layer's first group: the activations of the layer before are in shared memory
                if (g == 0 || g == 2 || g == 4) ok = mbar_wait(aready, (uint32_t)((g >> 1) & 1), wait_limit);
                if (ok && g >= 2) ok = mbar_wait(tfree + 8 * (g & 1), (uint32_t)(((g >> 1) - 1) & 1), wait_limit);
                for (int kc = 0; kc < 2 && ok; ++kc) {
                    const int c = 2 * g + kc;
                    ok = mbar_wait(wfull + 8 * (c % 3), (uint32_t)((c / 3) & 1), wait_limit);
                    if (ok) taken = c + 1;
                    if (!ok || idle) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    // descriptors differ in the start address alone (its 14 bits hold every address of
                    // the block): one add per operand
                    const uint32_t acc = tmem + (uint32_t)((g & 1) * TC);
                    const uint32_t w = wlo + (uint32_t)((c % 3) * (TILE_BYTES >> 4));
                    const uint32_t x = xlo + (uint32_t)((kc * (KC / 8) * (int)X_LBO) >> 4);
#pragma unroll
                    for (int s = 0; s < KC / 16; ++s)
                        mma(acc, desc_at(w + (uint32_t)((s * 2 * (int)W_LBO) >> 4), whi),
                            desc_at(x + (uint32_t)((s * 2 * (int)X_LBO) >> 4), xhi), IDESC, (kc | s) != 0);
                    commit(wfree + 8 * (c % 3));
                    // the chunk before is done with: its buffer takes the chunk after the next
                    if (c >= 1 && loaded < NCHUNK) {
                        ok = mbar_wait(wfree + 8 * ((c - 1) % 3), (uint32_t)(((c - 1) / 3) & 1), wait_limit);
                        if (ok) load();
                    }
                }
                if (ok) commit(mdone + 8 * (g & 1));
            }
            // copies still in flight land before the block leaves
            for (int i = taken; i < loaded; ++i) mbar_wait(wfull + 8 * (i % 3), (uint32_t)((i / 3) & 1), WAIT_LIMIT);
        }
    } else {
        // this thread: output f of every group, samples r0 .. r0 + 15 of the block
        const int f = 32 * (warp & 3) + lane, r0 = 16 * (warp >> 2);
        const int left = M - (m0 + r0);   // samples of them that exist
        const uint32_t tlane = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)r0;
        float v[2][16];   // a layer's activations of the thread's two outputs
        // bias and GELU of group c's sums, stored for the backward pass when training
        auto gelu_group = [&](int c, const float* bias, float* z, float* a) {
            const int o = TO * c + f;
            const float bb = bias[o];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float zz = v[c][i] + bb;
                v[c][i] = gelu_f(zz);
                if (TRAIN && i < left) {
                    const int64_t e = (int64_t)(m0 + r0 + i) * NH + o;
                    z[e] = zz;
                    a[e] = v[c][i];
                }
            }
        };
        // the layer's activations split into their three terms, to shared memory: 8 samples at once
        auto put = [&]() {
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float e[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) e[i] = v[c][8 * h + i];
#pragma unroll
                    for (int p = 0; p < TERMS; ++p) {
                        uint32_t t[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            t[i] = pack2(e[2 * i], e[2 * i + 1]);
                            e[2 * i] -= __uint_as_float(t[i] << 16);
                            e[2 * i + 1] -= __uint_as_float(t[i] & 0xffff0000u);
                        }
                        *reinterpret_cast<uint4*>(sm + x_off(TO * c + f, r0 + 8 * h, p)) = make_uint4(t[0], t[1], t[2], t[3]);
                    }
                }
            fence_smem_async();
            mbar_arrive(aready);
        };
        // layer 1: three inputs, on the CUDA cores
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float* w = fc + FC_W1 + (TO * c + f) * NIN;
            const float w0 = w[0], w1 = w[1], w2 = w[2];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float* x = fc + FC_X + (r0 + i) * NIN;
                v[c][i] = fmaf(x[2], w2, fmaf(x[1], w1, x[0] * w0));
            }
            gelu_group(c, fc + FC_B, tr.z[0], tr.a[0]);
        }
        put();
        int q = 0;
        auto take = [&](float (&t)[16]) {   // group q's sums
            ok = ok && mbar_wait(mdone + 8 * (q & 1), (uint32_t)((q >> 1) & 1), wait_limit);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) return;
            fence_after();
            // the three terms' sums, the smallest first
            const uint32_t acc = tlane + (uint32_t)((q & 1) * TC);
            float m[16], l[16];
            tmem_ld16(acc + 2 * TR, l);
            tmem_ld16(acc + TR, m);
            tmem_ld16(acc, t);
#pragma unroll
            for (int i = 0; i < 16; ++i) t[i] += m[i] + l[i];
            fence_before();
            mbar_arrive(tfree + 8 * (q & 1));
            ++q;
        };
#pragma unroll
        for (int l = 1; l < 3; ++l) {
            if (!ok) break;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if (!ok) break;
                take(v[c]);
                if (!ok) break;
                gelu_group(c, fc + FC_B + l * NH, tr.z[l], tr.a[l]);
            }
            if (ok) put();   // the layer's last MMA is done: its inputs may go
        }
        for (int c = 0; c < 4 && ok; ++c) {
            float t[16];
            take(t);
            const int o = TO * c + f;
            if (!ok || o >= NOUT) continue;
            const float bb = fc[FC_B + 3 * NH + o], sh = fc[FC_OUT + o], sc = fc[FC_OUT + NOUT + o];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                float y = t[i] + bb;
                if (!TRAIN) y = y * sc + sh;
                if (i < left) Y[(int64_t)(m0 + r0 + i) * NOUT + o] = y;
            }
        }
    }
    fence_before();
    ok = __syncthreads_and(ok);
    if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
    if (!ok && tid == 0) atomicExch(fault, 1);
}

template <bool TRAIN>
abs_status network_forward(abs_mlp* net, cudaStream_t st, const float* X, int64_t n, float* Y, bool idle = false) {
    MCK(cudaFuncSetAttribute(network_forward_kernel<TRAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, FWD_SMEM));
    FwdTrain tr{};
    if (TRAIN) {
        tr.a0 = net->a0;
        for (int l = 0; l < 3; ++l) {
            tr.z[l] = net->z[l];
            tr.a[l] = net->a[l];
        }
    }
    network_forward_kernel<TRAIN><<<(unsigned)((n + umma::TR - 1) / umma::TR), FWD_T, FWD_SMEM, st>>>(
        (int)n, X, net->norm, net->theta, net->wb, net->wt, Y, tr, net->dfault, idle ? 1 : 0,
        idle ? 1024ll : umma::WAIT_LIMIT);
    return mlaunch(net);
}

__global__ void normalize_kernel(int64_t n, const float* __restrict__ X, const float* __restrict__ norm,
                                 float* __restrict__ a0) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * NIN) return;
    const int k = (int)(i % NIN);
    a0[i] = (X[i] - norm[k]) / norm[NIN + k];
}

// g = (yhat - t) / (n * 440) with t the normalised target; block partial sums of r^2
__global__ void __launch_bounds__(256) loss_grad_kernel(int64_t n, const float* __restrict__ yh,
                                                        const float* __restrict__ Y, const float* __restrict__ norm,
                                                        float inv, float* __restrict__ g, double* __restrict__ part) {
    __shared__ double sh[256];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double r2 = 0.0;
    if (i < n * NOUT) {
        const int k = (int)(i % NOUT);
        const float t = (Y[i] - norm[2 * NIN + k]) / norm[2 * NIN + NOUT + k];
        const float r = yh[i] - t;
        g[i] = r * inv;
        r2 = (double)r * (double)r;
    }
    sh[threadIdx.x] = r2;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// out[slot] (+)= scale * sum of part[0..np) in a fixed order (one block)
__global__ void __launch_bounds__(256) sum_partials_kernel(const double* __restrict__ part, int64_t np, double scale,
                                                           bool accumulate, double* __restrict__ out) {
    __shared__ double sh[256];
    double a = 0.0;
    for (int64_t i = threadIdx.x; i < np; i += 256) a += part[i];
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = (accumulate ? *out : 0.0) + scale * sh[0];
}

// One layer of the backward pass in one launch: dW[o][i] = sum_r D[r][o] A[r][i], db[o] = sum_r
// D[r][o] and, in the remaining blocks, Dn[r][i] = (sum_o D[r][o] W[o][i]) gelu'(z[r][i]);
// D [n][O], A and z [n][I], W bfloat16 [O][I]; O and I multiples of 4, rows 16-byte aligned.  The
// products are independent: the first blocks take the 32 x 32 tiles of dW (those of the first column
// also db), the others the tiles of Dn.  A minibatch has few tiles for 152 SMs and a tile's
// sum is one chain of latencies, so the tiles are small and two groups of 128 threads share a tile's sum
// (even and odd steps of 32 terms, added at the end), each with the next step's global loads in
// flight while the current one is multiplied, 2 x 4 outputs per thread.  512 samples: 14.5 us per
// layer (strided GEMMs with 8 to 56 blocks and one-thread column sums: about 120).
constexpr int BT = 32, BT_G = 128;
constexpr int BT_SA = BT + 2, BT_SB = BT + 4;   // shared row strides: two-way conflicts at most on A's transposed stores
__global__ void __launch_bounds__(2 * BT_G) layer_backward_kernel(int n, int O, int I, const float* __restrict__ D,
                                                                  const float* __restrict__ A,
                                                                  const __nv_bfloat16* __restrict__ W,
                                                                  const float* __restrict__ z, float* __restrict__ dW,
                                                                  float* __restrict__ db, float* __restrict__ Dn) {
    __shared__ __align__(16) float As[2][2][BT][BT_SA];   // [group][buffer][k][m]
    __shared__ __align__(16) float Bs[2][2][BT][BT_SB];   // [group][buffer][k][n]
    const int grp = threadIdx.x / BT_G, tid = threadIdx.x % BT_G;
    const int tn = (I + BT - 1) / BT;
    const int tw = ((O + BT - 1) / BT) * tn;
    const bool isw = (int)blockIdx.x < tw;
    const int tile = isw ? blockIdx.x : blockIdx.x - tw;
    const int m0 = (tile / tn) * BT, n0 = (tile % tn) * BT;
    const int M = isw ? O : n, K = isw ? n : O;
    // four consecutive entries of rows hi and hi + 16 of a step's two tiles; D is read along its rows in
    // both products: D[k][m] for dW (hi = k, lo = m), D[m][k] for Dn (hi = m, lo = k)
    const int hi = tid >> 3, lo = (tid & 7) * 4;
    float4 ra[2], rb[2];
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int h = hi + 16 * q;
            const int kr = isw ? k0 + h : m0 + h, kc = isw ? m0 + lo : k0 + lo;   // D's row and column
            ra[q] = (kr < n && kc < O) ? *reinterpret_cast<const float4*>(D + (int64_t)kr * O + kc) : zero;
            rb[q] = zero;
            if (k0 + h < K && n0 + lo < I) {
                const int64_t e = (int64_t)(k0 + h) * I + n0 + lo;
                if (isw) {
                    rb[q] = *reinterpret_cast<const float4*>(A + e);
                } else {
                    const uint2 w = *reinterpret_cast<const uint2*>(W + e);   // four bfloat16
                    rb[q] = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                                        __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
                }
            }
        }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int h = hi + 16 * q;
            if (isw) {
                *reinterpret_cast<float2*>(&As[grp][b][h][lo]) = make_float2(ra[q].x, ra[q].y);
                *reinterpret_cast<float2*>(&As[grp][b][h][lo + 2]) = make_float2(ra[q].z, ra[q].w);
            } else {
                As[grp][b][lo][h] = ra[q].x;
                As[grp][b][lo + 1][h] = ra[q].y;
                As[grp][b][lo + 2][h] = ra[q].z;
                As[grp][b][lo + 3][h] = ra[q].w;
            }
            *reinterpret_cast<float4*>(&Bs[grp][b][h][lo]) = rb[q];
        }
    };
    const int tr = (tid >> 3) * 2, tc = (tid & 7) * 4;   // this thread's 2 rows and 4 columns
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    float colsum = 0.0f;
    const bool sums = isw && n0 == 0 && tid < BT;
    load(grp * BT);
    int b = 0;
    for (int k0 = grp * BT; k0 < K; k0 += 2 * BT, b ^= 1) {
        store(b);
        // one barrier of the group per step: the other buffer is free once all passed the last
        asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "r"(BT_G) : "memory");
        if (k0 + 2 * BT < K) load(k0 + 2 * BT);
#pragma unroll
        for (int k = 0; k < BT; ++k) {
            const float2 av = *reinterpret_cast<const float2*>(&As[grp][b][k][tr]);
            const float4 bv = *reinterpret_cast<const float4*>(&Bs[grp][b][k][tc]);
            const float br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc[0][j] = fmaf(av.x, br[j], acc[0][j]);
                acc[1][j] = fmaf(av.y, br[j], acc[1][j]);
            }
        }
        if (sums)
#pragma unroll
            for (int k = 0; k < BT; ++k) colsum += As[grp][b][k][tid];
    }
    __syncthreads();
    // the second group's sums, through its own tiles
    float* ex = &Bs[1][0][0][0];
    static_assert(2 * BT * BT_SB >= 9 * BT_G, "exchange fits");
    if (grp == 1) {
#pragma unroll
        for (int e = 0; e < 8; ++e) ex[e * BT_G + tid] = acc[e >> 2][e & 3];
        if (tid < BT) ex[8 * BT_G + tid] = colsum;
    }
    __syncthreads();
    if (grp == 1) return;
    if (sums && m0 + tid < O) db[m0 + tid] = colsum + ex[8 * BT_G + tid];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int m = m0 + tr + i;
        if (m >= M || n0 + tc >= I) continue;
        float o4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) o4[j] = acc[i][j] + ex[(4 * i + j) * BT_G + tid];
        const int64_t o = (int64_t)m * I + n0 + tc;
        if (!isw) {
            const float4 zz = *reinterpret_cast<const float4*>(z + o);
            o4[0] *= gelu_prime_f(zz.x);
            o4[1] *= gelu_prime_f(zz.y);
            o4[2] *= gelu_prime_f(zz.z);
            o4[3] *= gelu_prime_f(zz.w);
        }
        *reinterpret_cast<float4*>((isw ? dW : Dn) + o) = make_float4(o4[0], o4[1], o4[2], o4[3]);
    }
}

// the first layer's: dW[o][k] = sum_r D[r][o] a0[r][k] (three inputs), db[o] = sum_r D[r][o].  32 outputs
// per block on the lanes, the rows dealt to 32 warps, their sums added in warp order.
__global__ void __launch_bounds__(1024) first_backward_kernel(int n, const float* __restrict__ D,
                                                              const float* __restrict__ a0, float* __restrict__ dW,
                                                              float* __restrict__ db) {
    __shared__ float sm[4][32][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, o = blockIdx.x * 32 + lane;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int r = w; r < n; r += 32) {
        const float d = D[(int64_t)r * NH + o];
#pragma unroll
        for (int k = 0; k < NIN; ++k) s[k] = fmaf(d, a0[(int64_t)r * NIN + k], s[k]);
        s[3] += d;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) sm[k][w][lane] = s[k];
    __syncthreads();
    if (w >= 4) return;
    float t = 0.0f;
    for (int q = 0; q < 32; ++q) t += sm[w][q][lane];
    if (w < NIN) dW[(int64_t)o * NIN + w] = t;
    else db[o] = t;
}

// the rounded parameters, and the weights of layers 2-4 again in tiles
__device__ __forceinline__ void put_bf16(int64_t i, float v, __nv_bfloat16* wb, __nv_bfloat16* wt) {
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    wb[i] = h;
    const int t = tile_index(i);
    if (t >= 0) wt[t] = h;
}

// (and zeros for W4's outputs past the last)
__global__ void to_bf16_kernel(int64_t n, const float* __restrict__ src, __nv_bfloat16* __restrict__ wb,
                               __nv_bfloat16* __restrict__ wt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) put_bf16(i, src[i], wb, wt);
    constexpr int END = 4 * umma::TO;   // outputs the groups of W4 hold
    if (i < (END - NOUT) * NH) wt[tile_element(3, NOUT + (int)(i / NH), (int)(i % NH))] = __float2bfloat16_rn(0.0f);
}

__global__ void adam_kernel(int64_t n, float* __restrict__ th, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2,
                            __nv_bfloat16* __restrict__ wb, __nv_bfloat16* __restrict__ wt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float t = th[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    th[i] = t;
    put_bf16(i, t, wb, wt);
}

__global__ void gather_rows_kernel(int64_t rows, int cols, const int* __restrict__ idx, const float* __restrict__ src,
                                   float* __restrict__ dst) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * cols) return;
    const int64_t r = i / cols, c = i % cols;
    dst[i] = src[(int64_t)idx[r] * cols + c];
}

// per-column mean and standard deviation of X [n][cols] (double sums in a fixed order);
// a column whose spread is below 1e-7 of its magnitude keeps scale 1
__global__ void __launch_bounds__(256) column_stats_kernel(int64_t n, int cols, const float* __restrict__ X,
                                                           float* __restrict__ shift, float* __restrict__ scale) {
    __shared__ double sh[256];
    const int c = blockIdx.x;
    double a = 0.0;
    for (int64_t r = threadIdx.x; r < n; r += 256) a += X[r * cols + c];
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    const double mean = sh[0] / (double)n;
    __syncthreads();
    a = 0.0;
    for (int64_t r = threadIdx.x; r < n; r += 256) {
        const double d = X[r * cols + c] - mean;
        a += d * d;
    }
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double sd = sqrt(sh[0] / (double)n);
        shift[c] = (float)mean;
        scale[c] = (sd > 1e-7 * fmax(1.0, fabs(mean))) ? (float)sd : 1.0f;
    }
}

unsigned grid1(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

abs_status ensure_cap(abs_mlp* net, int64_t rows) {
    if (rows <= net->cap) return ABS_OK;
    cudaFree(net->a0);
    for (int l = 0; l < 3; ++l) {
        cudaFree(net->z[l]);
        cudaFree(net->a[l]);
    }
    cudaFree(net->yh);
    cudaFree(net->g);
    cudaFree(net->da);
    cudaFree(net->dz);
    cudaFree(net->xb);
    cudaFree(net->ybt);
    cudaFree(net->lpart);
    net->cap = 0;
    MCK(cudaMalloc(&net->a0, sizeof(float) * rows * NIN));
    for (int l = 0; l < 3; ++l) {
        MCK(cudaMalloc(&net->z[l], sizeof(float) * rows * NH));
        MCK(cudaMalloc(&net->a[l], sizeof(float) * rows * NH));
    }
    MCK(cudaMalloc(&net->yh, sizeof(float) * rows * NOUT));
    MCK(cudaMalloc(&net->g, sizeof(float) * rows * NOUT));
    MCK(cudaMalloc(&net->da, sizeof(float) * rows * NH));
    MCK(cudaMalloc(&net->dz, sizeof(float) * rows * NH));
    MCK(cudaMalloc(&net->xb, sizeof(float) * rows * NIN));
    MCK(cudaMalloc(&net->ybt, sizeof(float) * rows * NOUT));
    net->lpart_cap = (rows * NOUT + 255) / 256;
    MCK(cudaMalloc(&net->lpart, sizeof(double) * net->lpart_cap));
    net->cap = rows;
    return ABS_OK;
}

// forward pass of rows X [n][3] (raw); train: normalised outputs in net->yh and the
// layer values kept for backward; else raw outputs into Yout
abs_status forward_rows(abs_mlp* net, const float* X, int64_t n, bool train, float* Yout, cudaStream_t st) {
    if (net->tc) return train ? network_forward<true>(net, st, X, n, net->yh) : network_forward<false>(net, st, X, n, Yout);
    abs_status r;
    normalize_kernel<<<grid1(n * NIN), 256, 0, st>>>(n, X, net->norm, net->a0);
    if ((r = mlaunch(net)) != ABS_OK) return r;
    const float* prev = net->a0;
    for (int l = 0; l < 3; ++l) {
        if ((r = gemm<EPI_BIAS_GELU>(net, st, (int)n, NH, l_in(l), prev, net->wb + off_w(l), net->a[l],
                                     net->theta + off_b(l), net->z[l])) != ABS_OK)
            return r;
        prev = net->a[l];
    }
    if (train)
        return gemm<EPI_BIAS>(net, st, (int)n, NOUT, NH, prev, net->wb + off_w(3), net->yh, net->theta + off_b(3));
    return gemm<EPI_DENORM>(net, st, (int)n, NOUT, NH, prev, net->wb + off_w(3), Yout, net->theta + off_b(3), nullptr,
                            net->norm + 2 * NIN + NOUT, net->norm + 2 * NIN);
}

// loss and gradient of the rows last passed through forward_rows(train) against raw
// targets Y [n][440]; gradient into net->grad, loss*scale into *loss_dev (+= if acc)
abs_status backward_rows(abs_mlp* net, const float* Y, int64_t n, double* loss_dev, double scale, bool acc,
                         cudaStream_t st) {
    abs_status r;
    const int64_t nel = n * NOUT;
    const unsigned nb = grid1(nel);
    loss_grad_kernel<<<nb, 256, 0, st>>>(n, net->yh, Y, net->norm, 1.0f / (float)nel, net->g, net->lpart);
    if ((r = mlaunch(net)) != ABS_OK) return r;
    sum_partials_kernel<<<1, 256, 0, st>>>(net->lpart, nb, scale / (2.0 * (double)nel), acc, loss_dev);
    if ((r = mlaunch(net)) != ABS_OK) return r;
    // layer l: dW_l = dcur^T a_{l-1}, db_l = colsum dcur, dz_{l-1} = (dcur W_l) * gelu'(z_{l-1}); dcur
    // and the result alternate buffers
    const float* dcur = net->g;
    int ocur = NOUT;
    for (int l = 3; l > 0; --l) {
        float* dst = (dcur == net->dz) ? net->da : net->dz;
        const int64_t ti = NH / BT, tiles = ((ocur + BT - 1) / BT + (n + BT - 1) / BT) * ti;
        layer_backward_kernel<<<(unsigned)tiles, 2 * BT_G, 0, st>>>((int)n, ocur, NH, dcur, net->a[l - 1],
                                                                   net->wb + off_w(l), net->z[l - 1],
                                                                   net->grad + off_w(l), net->grad + off_b(l), dst);
        if ((r = mlaunch(net)) != ABS_OK) return r;
        dcur = dst;
        ocur = NH;
    }
    first_backward_kernel<<<NH / 32, 1024, 0, st>>>((int)n, dcur, net->a0, net->grad + off_w(0), net->grad + off_b(0));
    return mlaunch(net);
}

uint64_t splitmix64(uint64_t& s) {
    // splitmix64 (Steele, Lea & Flood 2014)
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

abs_status upload_norm(abs_mlp* net) {
    float f[2 * NIN + 2 * NOUT];
    for (int i = 0; i < 2 * NIN + 2 * NOUT; ++i) f[i] = (float)net->hnorm[i];
    MCK(cudaMemcpy(net->norm, f, sizeof(f), cudaMemcpyHostToDevice));
    return ABS_OK;
}

}  // namespace

extern "C" {

const char* abs_mlp_last_error(const abs_mlp* net) { return net ? net->err.c_str() : g_mlp_err.c_str(); }

abs_status abs_mlp_create(uint64_t seed, abs_mlp** out) {
    abs_mlp* net = nullptr;
    if (!out) return mfail(nullptr, ABS_ERR_ARG, "bad argument");
    *out = nullptr;
    net = new abs_mlp();
    abs_status r = ABS_OK;
    auto bad = [&](abs_status st) {
        const std::string msg = net->err;
        abs_mlp_destroy(net);
        return mfail(nullptr, st, msg);
    };
#define MCK2(call)                                                                                    \
    do {                                                                                              \
        cudaError_t e_ = (call);                                                                      \
        if (e_ != cudaSuccess) {                                                                      \
            mfail(net, e_ == cudaErrorMemoryAllocation ? ABS_ERR_OOM : ABS_ERR_CUDA,                  \
                  std::string(#call) + ": " + cudaGetErrorString(e_));                                \
            return bad(e_ == cudaErrorMemoryAllocation ? ABS_ERR_OOM : ABS_ERR_CUDA);                 \
        }                                                                                             \
    } while (0)
    MCK2(cudaGetDevice(&net->dev));
    // one allocation: theta, grad, m, v, norm (floats), then wb, wt (bfloat16); every part 256-byte aligned
    constexpr size_t PF = (NPAR + 63) / 64 * 64, PN = (2 * NIN + 2 * NOUT + 63) / 64 * 64, PB = (NPAR + 127) / 128 * 128;
    MCK2(cudaMalloc(&net->theta, sizeof(float) * (4 * PF + PN) + sizeof(__nv_bfloat16) * (PB + NCHUNK * CHUNK_ELS)));
    net->grad = net->theta + PF;
    net->m = net->grad + PF;
    net->v = net->m + PF;
    net->norm = net->v + PF;
    net->wb = reinterpret_cast<__nv_bfloat16*>(net->norm + PN);
    net->wt = net->wb + PB;
    MCK2(cudaHostAlloc(&net->hfault, sizeof(int), cudaHostAllocMapped));
    *net->hfault = 0;
    MCK2(cudaHostGetDevicePointer(&net->dfault, net->hfault, 0));
#undef MCK2
    // Glorot-uniform weights (Glorot & Bengio 2010), zero biases, identity normalisation
    std::vector<float> th(NPAR, 0.0f);
    uint64_t s = seed;
    for (int l = 0; l < 4; ++l) {
        const double lim = std::sqrt(6.0 / (double)(l_in(l) + l_out(l)));
        for (int64_t i = 0; i < (int64_t)l_in(l) * l_out(l); ++i) {
            const double u = (double)(splitmix64(s) >> 11) * (1.0 / 9007199254740992.0);
            th[off_w(l) + i] = (float)((2.0 * u - 1.0) * lim);
        }
    }
    for (int i = 0; i < NIN; ++i) {
        net->hnorm[i] = 0.0;
        net->hnorm[NIN + i] = 1.0;
    }
    for (int i = 0; i < NOUT; ++i) {
        net->hnorm[2 * NIN + i] = 0.0;
        net->hnorm[2 * NIN + NOUT + i] = 1.0;
    }
    if ((r = upload_norm(net)) != ABS_OK) return bad(r);
    if ((r = abs_mlp_set_params(net, th.data())) != ABS_OK) return bad(r);
    *out = net;
    return ABS_OK;
}

void abs_mlp_destroy(abs_mlp* net) {
    if (!net) return;
    if (net->hfault) cudaFreeHost(net->hfault);
    cudaFree(net->theta);   // with grad, m, v, norm, wb, wt
    cudaFree(net->a0);
    for (int l = 0; l < 3; ++l) {
        cudaFree(net->z[l]);
        cudaFree(net->a[l]);
    }
    cudaFree(net->yh);
    cudaFree(net->g);
    cudaFree(net->da);
    cudaFree(net->dz);
    cudaFree(net->xb);
    cudaFree(net->ybt);
    cudaFree(net->perm);
    cudaFree(net->lpart);
    cudaFree(net->lacc);
    delete net;
}

abs_status abs_mlp_set_params(abs_mlp* net, const float* params) {
    if (!net || !params) return mfail(net, ABS_ERR_ARG, "bad argument");
    MCK(cudaMemcpy(net->theta, params, sizeof(float) * NPAR, cudaMemcpyHostToDevice));
    MCK(cudaMemset(net->m, 0, (size_t)((char*)(net->v + NPAR) - (char*)net->m)));   // both moments
    net->step = 0;
    to_bf16_kernel<<<grid1(NPAR), 256>>>(NPAR, net->theta, net->wb, net->wt);
    abs_status r = mlaunch(net);
    if (r != ABS_OK) return r;
    MCK(cudaDeviceSynchronize());
    return ABS_OK;
}

abs_status abs_mlp_get_params(const abs_mlp* cnet, float* params) {
    abs_mlp* net = const_cast<abs_mlp*>(cnet);
    if (!net || !params) return mfail(net, ABS_ERR_ARG, "bad argument");
    MCK(cudaMemcpy(params, net->theta, sizeof(float) * NPAR, cudaMemcpyDeviceToHost));
    return ABS_OK;
}

abs_status abs_mlp_set_normalization(abs_mlp* net, const double* in_shift, const double* in_scale,
                                     const double* out_shift, const double* out_scale) {
    if (!net || !in_shift || !in_scale || !out_shift || !out_scale) return mfail(net, ABS_ERR_ARG, "bad argument");
    for (int i = 0; i < NIN; ++i)
        if (!(in_scale[i] > 0.0)) return mfail(net, ABS_ERR_ARG, "scales must be positive");
    for (int i = 0; i < NOUT; ++i)
        if (!(out_scale[i] > 0.0)) return mfail(net, ABS_ERR_ARG, "scales must be positive");
    std::memcpy(net->hnorm, in_shift, sizeof(double) * NIN);
    std::memcpy(net->hnorm + NIN, in_scale, sizeof(double) * NIN);
    std::memcpy(net->hnorm + 2 * NIN, out_shift, sizeof(double) * NOUT);
    std::memcpy(net->hnorm + 2 * NIN + NOUT, out_scale, sizeof(double) * NOUT);
    return upload_norm(net);
}

abs_status abs_mlp_get_normalization(const abs_mlp* net, double* in_shift, double* in_scale, double* out_shift,
                                     double* out_scale) {
    if (!net) return mfail(nullptr, ABS_ERR_ARG, "bad argument");
    if (in_shift) std::memcpy(in_shift, net->hnorm, sizeof(double) * NIN);
    if (in_scale) std::memcpy(in_scale, net->hnorm + NIN, sizeof(double) * NIN);
    if (out_shift) std::memcpy(out_shift, net->hnorm + 2 * NIN, sizeof(double) * NOUT);
    if (out_scale) std::memcpy(out_scale, net->hnorm + 2 * NIN + NOUT, sizeof(double) * NOUT);
    return ABS_OK;
}

abs_status abs_mlp_fit_normalization(abs_mlp* net, const float* X, const float* Y, int64_t n, abs_stream_t stream) {
    if (!net || !X || !Y || n < 1) return mfail(net, ABS_ERR_ARG, "bad argument");
    cudaStream_t st = (cudaStream_t)stream;
    column_stats_kernel<<<NIN, 256, 0, st>>>(n, NIN, X, net->norm, net->norm + NIN);
    abs_status r = mlaunch(net);
    if (r != ABS_OK) return r;
    column_stats_kernel<<<NOUT, 256, 0, st>>>(n, NOUT, Y, net->norm + 2 * NIN, net->norm + 2 * NIN + NOUT);
    if ((r = mlaunch(net)) != ABS_OK) return r;
    float f[2 * NIN + 2 * NOUT];
    MCK(cudaMemcpyAsync(f, net->norm, sizeof(f), cudaMemcpyDeviceToHost, st));
    MCK(cudaStreamSynchronize(st));
    for (int i = 0; i < 2 * NIN + 2 * NOUT; ++i) net->hnorm[i] = f[i];
    return ABS_OK;
}

int32_t abs_mlp_device_fault(const abs_mlp* net) { return net && net->hfault ? *(volatile int*)net->hfault : 0; }

abs_status abs_mlp_set_tensor_cores(abs_mlp* net, int32_t on) {
    if (!net || (on != 0 && on != 1)) return mfail(net, ABS_ERR_ARG, "bad argument");
    net->tc = on != 0;
    return ABS_OK;
}

abs_status abs_mlp_selftest_wait(abs_mlp* net, abs_stream_t stream) {
    if (!net) return mfail(net, ABS_ERR_ARG, "bad argument");
    if (abs_mlp_device_fault(net)) return mfail(net, ABS_ERR_TIMEOUT, "a tensor-core product gave up waiting");
    cudaStream_t st = (cudaStream_t)stream;
    abs_status r;
    if ((r = ensure_cap(net, umma::TR)) != ABS_OK) return r;
    // one block's forward pass with its MMAs withheld, on the activation workspace
    MCK(cudaMemsetAsync(net->xb, 0, sizeof(float) * umma::TR * NIN, st));
    if ((r = network_forward<true>(net, st, net->xb, umma::TR, net->yh, true)) != ABS_OK) return r;
    MCK(cudaStreamSynchronize(st));
    const bool expired = abs_mlp_device_fault(net) != 0;
    *(volatile int*)net->hfault = 0;
    if (!expired) return mfail(net, ABS_ERR_CUDA, "the withheld wait did not report its expiry");
    return mfail(net, ABS_ERR_TIMEOUT, "a tensor-core product gave up waiting (self-test)");
}

abs_status abs_mlp_forward(abs_mlp* net, const float* X, int64_t n, float* Y, abs_stream_t stream) {
    if (!net || n < 0 || (n > 0 && (!X || !Y))) return mfail(net, ABS_ERR_ARG, "bad argument");
    if (abs_mlp_device_fault(net)) return mfail(net, ABS_ERR_TIMEOUT, "a tensor-core product gave up waiting");
    cudaStream_t st = (cudaStream_t)stream;
    abs_status r;
    if (n == 0) return ABS_OK;
    // the tensor-core pass keeps its activations on chip: no workspace, any number of rows (in pieces a
    // launch's row index holds)
    const int64_t piece = net->tc ? (int64_t)1 << 30 : CHUNK_ROWS;
    for (int64_t r0 = 0; r0 < n; r0 += piece) {
        const int64_t rows = std::min<int64_t>(piece, n - r0);
        if (!net->tc && (r = ensure_cap(net, rows)) != ABS_OK) return r;
        if ((r = forward_rows(net, X + r0 * NIN, rows, false, Y + r0 * NOUT, st)) != ABS_OK) return r;
    }
    return ABS_OK;
}

abs_status abs_mlp_loss_grad(abs_mlp* net, const float* X, const float* Y, int64_t n, double* loss, float* grad,
                             abs_stream_t stream) {
    if (!net || !X || !Y || n < 1) return mfail(net, ABS_ERR_ARG, "bad argument");
    if (abs_mlp_device_fault(net)) return mfail(net, ABS_ERR_TIMEOUT, "a tensor-core product gave up waiting");
    cudaStream_t st = (cudaStream_t)stream;
    abs_status r;
    if ((r = ensure_cap(net, n)) != ABS_OK) return r;
    if (!net->lacc) {
        MCK(cudaMalloc(&net->lacc, sizeof(double) * 64));
        net->lacc_cap = 64;
    }
    if ((r = forward_rows(net, X, n, true, nullptr, st)) != ABS_OK) return r;
    if ((r = backward_rows(net, Y, n, net->lacc, 1.0, false, st)) != ABS_OK) return r;
    if (grad) MCK(cudaMemcpyAsync(grad, net->grad, sizeof(float) * NPAR, cudaMemcpyDeviceToDevice, st));
    double l = 0.0;
    MCK(cudaMemcpyAsync(&l, net->lacc, sizeof(double), cudaMemcpyDeviceToHost, st));
    MCK(cudaStreamSynchronize(st));
    if (loss) *loss = l;
    return ABS_OK;
}

void abs_default_train_options(abs_train_options* o) {
    if (!o) return;
    std::memset(o, 0, sizeof(*o));
    o->epochs = 200;
    o->batch = 512;
    o->lr = 1e-3;
    o->lr_final = 1e-5;
    o->beta1 = 0.9;
    o->beta2 = 0.999;
    o->eps = 1e-8;
    o->seed = 1;
}

abs_status abs_mlp_train(abs_mlp* net, const float* X, const float* Y, int64_t n, const abs_train_options* opt_in,
                         double* epoch_loss, abs_stream_t stream) {
    if (!net || !X || !Y || n < 1) return mfail(net, ABS_ERR_ARG, "bad argument");
    if (abs_mlp_device_fault(net)) return mfail(net, ABS_ERR_TIMEOUT, "a tensor-core product gave up waiting");
    abs_train_options o;
    if (opt_in) o = *opt_in;
    else abs_default_train_options(&o);
    if (o.epochs < 1 || o.batch < 1 || !(o.lr > 0) || !(o.lr_final > 0) || !(o.beta1 >= 0 && o.beta1 < 1) ||
        !(o.beta2 >= 0 && o.beta2 < 1) || !(o.eps > 0) || n > INT32_MAX)
        return mfail(net, ABS_ERR_ARG, "bad training option");
    cudaStream_t st = (cudaStream_t)stream;
    abs_status r;
    const int64_t B = std::min<int64_t>(o.batch, n);
    if ((r = ensure_cap(net, B)) != ABS_OK) return r;
    if (net->perm_cap < n) {
        cudaFree(net->perm);
        net->perm = nullptr;
        MCK(cudaMalloc(&net->perm, sizeof(int) * n));
        net->perm_cap = n;
    }
    if (net->lacc_cap < o.epochs) {
        cudaFree(net->lacc);
        net->lacc = nullptr;
        MCK(cudaMalloc(&net->lacc, sizeof(double) * o.epochs));
        net->lacc_cap = o.epochs;
    }
    std::vector<int> perm(n);
    uint64_t rs = o.seed;
    for (int e = 0; e < o.epochs; ++e) {
        // this epoch's order: Fisher-Yates shuffle with splitmix64 draws
        for (int64_t i = 0; i < n; ++i) perm[i] = (int)i;
        for (int64_t i = n - 1; i > 0; --i) {
            const int64_t j = (int64_t)(splitmix64(rs) % (uint64_t)(i + 1));
            std::swap(perm[i], perm[j]);
        }
        // the copy reads perm before this host loop writes it again (synchronised below)
        MCK(cudaMemcpyAsync(net->perm, perm.data(), sizeof(int) * n, cudaMemcpyHostToDevice, st));
        const double lr =
            o.epochs > 1 ? o.lr * std::pow(o.lr_final / o.lr, (double)e / (double)(o.epochs - 1)) : o.lr;
        bool first = true;
        for (int64_t b0 = 0; b0 < n; b0 += B) {
            const int64_t nb = std::min<int64_t>(B, n - b0);
            gather_rows_kernel<<<grid1(nb * NIN), 256, 0, st>>>(nb, NIN, net->perm + b0, X, net->xb);
            if ((r = mlaunch(net)) != ABS_OK) return r;
            gather_rows_kernel<<<grid1(nb * NOUT), 256, 0, st>>>(nb, NOUT, net->perm + b0, Y, net->ybt);
            if ((r = mlaunch(net)) != ABS_OK) return r;
            if ((r = forward_rows(net, net->xb, nb, true, nullptr, st)) != ABS_OK) return r;
            if ((r = backward_rows(net, net->ybt, nb, net->lacc + e, (double)nb / (double)n, !first, st)) != ABS_OK)
                return r;
            first = false;
            net->step++;
            const double c1 = 1.0 - std::pow(o.beta1, (double)net->step);
            const double c2 = 1.0 - std::pow(o.beta2, (double)net->step);
            adam_kernel<<<grid1(NPAR), 256, 0, st>>>(NPAR, net->theta, net->grad, net->m, net->v, (float)lr,
                                                     (float)o.beta1, (float)o.beta2, (float)o.eps, (float)c1,
                                                     (float)c2, net->wb, net->wt);
            if ((r = mlaunch(net)) != ABS_OK) return r;
        }
        MCK(cudaStreamSynchronize(st));
    }
    if (epoch_loss)
        MCK(cudaMemcpyAsync(epoch_loss, net->lacc, sizeof(double) * o.epochs, cudaMemcpyDeviceToHost, st));
    MCK(cudaStreamSynchronize(st));
    return ABS_OK;
}

}  // extern "C"
