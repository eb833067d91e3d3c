// kernels_umma.cuh -- tcgen05 (fifth-generation tensor core) building blocks of the warm-start
// network's forward pass (network_forward_kernel, mlp_lib.cu): kind::f16 MMAs on shared-memory
// operands in the no-swizzle core-matrix layouts, FP32 accumulators in tensor memory, mbarriers, bulk
// copies.
//
// An MMA takes both operands in one type and the weights are bfloat16, so each FP32 activation
// enters as the sum of three bfloat16 terms a = h + m + l (h the rounding of a, m of a - h, l of
// a - h - m: 24 significand bits); the three products with a bfloat16 weight are exact in the FP32
// accumulator.  The three terms of 64 samples stand side by side as 192 columns of one MMA, so a weight
// is read from shared memory once for all three: 24 MMAs of 64 columns took 1.6-2.1 k cycles per chunk of
// weights whatever their M, and 8 of 192 columns brought 5000 samples from 30.8 to 26.6 us.  An output's
// three sums are added as they leave tensor memory.
#pragma once

#include <cuda_bf16.h>
#include <cstdint>

namespace umma {

// A layer's products are formed transposed, outputs as the MMA's 128 rows and samples as its
// columns: 64 samples per block leave few SMs idle at 5000 samples, an accumulator lane is an output, so
// its bias is one register, and a lane stores eight samples of a term at once (samples as rows: 43 us).
constexpr int TR = 64, TK = 256;                  // samples of a block; a layer's inputs
constexpr int TO = 128, KC = 128;                 // outputs and inputs of a weight chunk
constexpr int TILE_BYTES = TO * KC * 2;           // a weight chunk
// Core matrices are 128 bytes.  Weights are K-major: 8 outputs x 8 inputs, an output's 8 inputs in 16
// bytes.  Activations are sample-major: 8 inputs x 8 samples, an input's 8 samples in 16 bytes (what a
// lane that holds one output for many samples stores at once).  Both: core matrices adjacent along
// outputs / samples 128 bytes apart ("stride"), along the inputs after them ("leading").
constexpr int TERMS = 3, TC = TERMS * TR;         // terms of an activation; an accumulator's columns
constexpr uint32_t SBO = 128, W_LBO = (TO / 8) * 128, X_LBO = (TC / 8) * 128;
constexpr int ACT_BYTES = TC * TK * 2;            // the activations
constexpr int TMEM_COLS = 512;                    // two accumulators of 192, a power of two
constexpr long long WAIT_LIMIT = 1ll << 22;       // mbarrier polls before a wait gives up

// instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B bfloat16 (bits 7-9,
// 10-12 = 1), A K-major (bit 15 = 0), B N-major (bit 16 = 1), N >> 3 at bit 17, M >> 4 at bit 24
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(TC >> 3) << 17) |
                           ((uint32_t)(TO >> 4) << 24);

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start address, leading / stride byte offsets (all >> 4),
// descriptor version 1 at bits 46-47, base offset 0, no swizzle
__device__ __forceinline__ uint64_t desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo & 0x3FFFFu) >> 4) << 16) |
           ((uint64_t)((sbo & 0x3FFFFu) >> 4) << 32) | (1ull << 46);
}

__device__ __forceinline__ uint64_t desc_at(uint32_t lo, uint32_t hi) { return ((uint64_t)hi << 32) | lo; }

__device__ __forceinline__ void tmem_alloc(uint32_t dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// the threads' shared-memory stores become visible to the tensor cores (async proxy)
__device__ __forceinline__ void fence_smem_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mma(uint32_t dt, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dt),
        "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate)
        : "memory");
}
// the mbarrier completes its phase when every MMA this thread issued so far is done
__device__ __forceinline__ void commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(mbar), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait for the completion of phase `parity` (at most `limit` polls); false when it
// gave up
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, long long limit) {
    for (long long it = 0; it < limit; ++it)
        if (mbar_try(mbar, parity)) return true;
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
// bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned) to shared memory; its
// arrival completes on mbar
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
        "r"(bytes), "r"(mbar)
        : "memory");
}

// 16 consecutive accumulator columns of this thread's lane (32x32b shape: lane = row)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// byte offset of weight (output o, input k) in a chunk; of term p of activation (input k, sample r)
__host__ __device__ constexpr uint32_t w_off(int o, int k) {
    return (uint32_t)((((k >> 3) * (TO / 8) + (o >> 3)) << 7) + ((o & 7) << 4) + ((k & 7) << 1));
}
__host__ __device__ constexpr uint32_t x_off(int k, int r, int p) {
    return (uint32_t)((((k >> 3) * (TC / 8) + p * (TR / 8) + (r >> 3)) << 7) + ((k & 7) << 4) + ((r & 7) << 1));
}

// two values rounded to bfloat16, the first in the low half
__device__ __forceinline__ uint32_t pack2(float a, float b) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
    return r;
}

}  // namespace umma
