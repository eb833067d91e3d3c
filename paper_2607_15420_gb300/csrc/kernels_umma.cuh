// kernels_umma.cuh -- tcgen05 (fifth-generation tensor core) building blocks of the warm-start
// network's forward pass (network_forward_kernel, mlp_lib.cu): kind::f16 MMAs on shared-memory
// operands in the no-swizzle K-major core-matrix layout, FP32 accumulators in tensor memory,
// mbarriers, bulk copies.
//
// An MMA takes both operands in one type and the weights are bfloat16, so each FP32 activation
// enters as the sum of three bfloat16 terms a = h + m + l (h the rounding of a, m of a - h, l of
// a - h - m: 24 significand bits); the three products with a bfloat16 weight are exact in the FP32
// accumulator: a layer's product at FP32 accuracy from three MMAs per K step.
#pragma once

#include <cuda_bf16.h>
#include <cstdint>

namespace umma {

constexpr int TM = 64, TN = 64, TK = 256;         // a block's rows; a weight chunk's columns; inputs
constexpr int TILE_BYTES = TM * TK * 2;           // one bfloat16 term of the activations; a weight chunk
// core matrices are 8 rows x 16 bytes; 8 row groups per 8-column K block: strides in bytes between core
// matrices adjacent along K ("leading") and along M / N ("stride")
constexpr uint32_t LBO = (TM / 8) * 128, SBO = 128;
constexpr long long WAIT_LIMIT = 1ll << 22;       // mbarrier polls before a wait gives up
static_assert(TM == TN, "activations and weight chunks share one layout");

// instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B bfloat16 (bits 7-9,
// 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bit 17, M >> 4 at bit 24
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start address, leading / stride byte offsets (all >> 4),
// descriptor version 1 at bits 46-47, base offset 0, no swizzle
__device__ __forceinline__ uint64_t desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo & 0x3FFFFu) >> 4) << 16) |
           ((uint64_t)((sbo & 0x3FFFFu) >> 4) << 32) | (1ull << 46);
}

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

// 16 accumulator columns of 16 rows over the warp (16x256b shape): thread t gets, for i < 2, columns 8 i
// + 2 (t % 4) + {0, 1} of row t / 4 in v[4 i + {0, 1}] and of row t / 4 + 8 in v[4 i + {2, 3}].  An M = 64
// accumulator keeps rows 16 w .. 16 w + 15 in the first 16 lanes of the 32 that warp w (mod 4) reads.
__device__ __forceinline__ void tmem_ld_16x16(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// byte offset of element (r, k) of a 64-row tile in core-matrix layout
__device__ __forceinline__ uint32_t core_off(int r, int k) {
    return (uint32_t)((((k >> 3) * (TM / 8) + (r >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1));
}

__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 a, __nv_bfloat16 b) {
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

}  // namespace umma
