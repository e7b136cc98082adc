// tc_ptx.cuh -- inline-PTX wrappers for the 5th-generation tensor cores
// (tcgen05: MMA, commit, tensor-memory loads), the tensor memory accelerator
// (cp.async.bulk.tensor) and mbarriers, shared by the projection GEMM
// (k_tc.cu) and the fused assembly-projection kernel (k_fused.cu).
// Every mbarrier wait is bounded (TC_WAIT_NS of wall clock).
#pragma once

#include <cuda.h>   // CUtensorMap
#include <stdint.h>

namespace cbfm {
namespace tc {

constexpr int TC_M = 128;                        // rows per MMA tile (M)
constexpr uint64_t TC_WAIT_NS = 1000000000ull;   // 1 s per wait

// ------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t gtimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase with the given parity to complete; false after TC_WAIT_NS.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    if (mbar_try(bar, parity)) return true;
    const uint64_t t0 = gtimer();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (gtimer() - t0 > TC_WAIT_NS) return false;
    }
}

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2,
                                            int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_u32(dst)),
        "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row
// groups 1024 bytes apart (stride byte offset), descriptor version 1.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024u >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Instruction descriptor, kind::tf32: D F32, A and B TF32, both K-major, M = 128.
__device__ __forceinline__ uint32_t idesc_tf32(int n) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t dtmem, uint64_t ad, uint64_t bd, uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(
            dtmem),
        "l"(ad), "l"(bd), "r"(id), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// TF32 rounding (round to nearest, ties away from zero), low 13 bits zero.
__device__ __forceinline__ float tf32r(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

__device__ __forceinline__ void split(float x, float &hi, float &lo) {
    hi = tf32r(x);
    lo = tf32r(x - hi);
}

__device__ __forceinline__ void split64(double x, float &hi, float &lo) {
    hi = tf32r((float)x);
    lo = tf32r((float)(x - (double)hi));
}


// 128-byte-swizzled K-major tile of 32 floats per row (the layout TMA writes
// with CU_TENSOR_MAP_SWIZZLE_128B and sdesc() describes): byte offset of float
// f (0..31) of row r from a 1024-byte-aligned tile base.
__device__ __forceinline__ uint32_t swz128(int r, int f) {
    return (uint32_t)r * 128u + ((((uint32_t)(f >> 2)) ^ ((uint32_t)r & 7u)) << 4) + ((uint32_t)(f & 3) << 2);
}

// 64-byte-swizzled K-major tile of 16 floats per row: byte offset of float f
// (0..15) of row r from a 512-byte-aligned tile base (16-byte chunk index XOR
// address bits 7-8, i.e. the row pair within the 8-row, 512-byte atom).
__device__ __forceinline__ uint32_t swz64(int r, int f) {
    return (uint32_t)r * 64u + ((((uint32_t)(f >> 2)) ^ (((uint32_t)r >> 1) & 3u)) << 4) + ((uint32_t)(f & 3) << 2);
}

// Shared-memory matrix descriptor for a K-major operand with the 64-byte
// swizzle: 8-row groups 512 bytes apart (stride byte offset), descriptor
// version 1, swizzle mode 4.
__device__ __forceinline__ uint64_t sdesc64(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512u >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

// The same with the 32-byte swizzle (8 floats per row, one K step): 16-byte chunk index XOR address bit 7,
// 8-row groups 256 bytes apart, swizzle mode 6.
__device__ __forceinline__ uint32_t swz32(int r, int f) {
    return (uint32_t)r * 32u + ((((uint32_t)(f >> 2)) ^ (((uint32_t)r >> 2) & 1u)) << 4) + ((uint32_t)(f & 3) << 2);
}
__device__ __forceinline__ uint64_t sdesc32(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(256u >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)6 << 61);
}

}  // namespace tc
}  // namespace cbfm
