// tc_ptx.cuh -- the tensor-core building blocks shared by m2l_tc.cu and m2l_oz.cu: swizzled operand
// layouts, matrix and instruction descriptors, bounded mbarrier waits, bulk copies and tcgen05
// wrappers (inline PTX for sm_103a).
#pragma once

#include <cuda.h>  // CUtensorMap and its enums; the encoder itself is looked up at run time
#include <cuda_bf16.h>
#include <stdint.h>

namespace {

constexpr int TC_M = 128;                    // real-form rows (2 p^2 <= 128)
constexpr int KBLK = 32;                     // TF32 elements per 128-byte swizzle row
constexpr int A_KB_BYTES = TC_M * KBLK * 4;  // 16 KiB of A per K block
constexpr int MAX_STAGES = 8;
constexpr int SMEM_BUDGET = 200 * 1024;      // dynamic shared memory for the stages
constexpr uint64_t WAIT_NS = 2000000000ull;  // a stage turns over in about a microsecond

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// float index of element (row, k) of one 128-row K block in the 128-byte-swizzled K-major layout:
// rows 128 bytes apart, the 16-byte chunk c of row m stored at chunk c ^ (m mod 8)
__host__ __device__ __forceinline__ int sw128_index(int row, int k) {
    return row * KBLK + (((k >> 2) ^ (row & 7)) << 2) + (k & 3);
}

// shared-memory matrix descriptor, K-major, 128-byte swizzle: 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;            // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;  // stride byte offset
    d |= (uint64_t)1 << 46;            // descriptor version of the sm_100 family
    d |= (uint64_t)2 << 61;            // 128-byte swizzle
    return d;
}

// instruction descriptor: D f32, A and B tf32, both K-major, M = 128, N = n
__host__ __device__ constexpr uint32_t idesc_tf32(int n) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}
// instruction descriptor of kind::f16: D f32, A and B bf16, both K-major, M = 128, N = n
__host__ __device__ constexpr uint32_t idesc_bf16(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}

// bf16 index of element (row, k) of one K block (32 bf16 = 64 bytes per row) in the 64-byte-swizzled
// K-major layout: the 16-byte chunk c of row m stored at chunk c ^ ((m / 2) mod 4)
__host__ __device__ __forceinline__ int sw64_index(int row, int k) {
    return row * KBLK + ((((k >> 3) ^ (row >> 1)) & 3) << 3) + (k & 7);
}

// shared-memory matrix descriptor, K-major, 64-byte swizzle: 8-row groups 512 bytes apart
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;           // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(512 >> 4) << 32;  // stride byte offset
    d |= (uint64_t)1 << 46;           // descriptor version of the sm_100 family
    d |= (uint64_t)4 << 61;           // 64-byte swizzle
    return d;
}

__device__ __forceinline__ float to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint64_t *m, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(m)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *m, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(m)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait for the phase of the given parity; false on time-out
__device__ __noinline__ bool mbar_wait(uint64_t *m, uint32_t parity) {
    if (mbar_try_wait(m, parity)) return true;
    const uint64_t t0 = globaltimer();
    for (;;) {
        for (int i = 0; i < 64; ++i)
            if (mbar_try_wait(m, parity)) return true;
        if (globaltimer() - t0 > WAIT_NS) return false;
    }
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *m, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(m)), "r"(bytes) : "memory");
}
// 1-D bulk copy global -> shared, completion counted on the mbarrier
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint64_t *m) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(smem_u32(m))
                 : "memory");
}
// 2-D tiled tensor copy global -> shared (box and swizzle from the tensor map)
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *tm, int x, int y, uint64_t *m) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(dst),
        "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(smem_u32(m))
        : "memory");
}
__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// the same for a whole warp of which one lane (issue != 0) issues; COLL: the A operand is read and
// dropped (0), read and kept in the collector (1), taken from it (2) or taken from it last (3)
template <int COLL>
__device__ __forceinline__ void mma_bf16_if(uint32_t issue, uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
#define FMBEM_MMA_IF(usage)                                                                                            \
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"                        \
                 "@q tcgen05.mma.cta_group::1.kind::f16" usage " [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),            \
                 "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(issue)                                        \
                 : "memory")
    if constexpr (COLL == 0) FMBEM_MMA_IF("");
    else if constexpr (COLL == 1) FMBEM_MMA_IF(".collector::a::fill");
    else if constexpr (COLL == 2) FMBEM_MMA_IF(".collector::a::use");
    else FMBEM_MMA_IF(".collector::a::lastuse");
#undef FMBEM_MMA_IF
}
__device__ __forceinline__ void mma_commit(uint64_t *m) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(m))
                 : "memory");
}

}  // namespace
