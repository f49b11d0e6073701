// Fifth-generation tensor-core helpers (tcgen05, sm_100 family): tensor-memory
// allocation, shared-memory operand descriptors, bf16 MMA with FP32
// accumulation in tensor memory, completion through an mbarrier, and loads of
// the accumulator back to registers.
//
// Operand layout: every MMA operand here is a [R rows][K] bf16 matrix in
// shared memory, K-major, without swizzling, stored as 8 x 8 "core matrices"
// of 128 contiguous bytes (row r of a core matrix at byte 16 r).  Core matrix
// (row group g, k chunk c) sits at byte 128 (g (K/8) + c), so the byte
// distance between core matrices adjacent in K (the leading-dimension offset)
// is 128 and between adjacent row groups (the stride-dimension offset) is
// 16 K.  One MMA consumes 16 values of K: two core-matrix columns.
#pragma once
#include <cstdint>

namespace vdw {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// element index of (r, k) in the K-major core-matrix layout of a K-wide operand
__device__ __forceinline__ int kmaj(int r, int k, int K) {
    return (((r >> 3) * (K >> 3) + (k >> 3)) << 6) + ((r & 7) << 3) + (k & 7);
}

// shared-memory matrix descriptor: start address, leading- and stride-dimension
// byte offsets (all in 16-byte units), descriptor version 1, no swizzling
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// descriptor of K-step s (16 values of K) of a K-wide operand starting at addr
__device__ __forceinline__ uint64_t operand_desc(uint32_t addr, int K, int s) {
    return smem_desc(addr + 256u * (uint32_t)s, 128u, 16u * (uint32_t)K);
}

// instruction descriptor: kind::f16 with bf16 A and B, FP32 accumulator,
// both operands K-major, M x N tile
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The same stored tile read the other way: a [R rows][K] tile as the operand
// whose M (or N) index is the tile's k and whose contraction runs over the
// tile's rows (MN-major, no swizzling: the stride-dimension offset is the
// distance of core matrices adjacent in M or N, the leading-dimension offset
// that of core matrices adjacent in the contraction).  Descriptor of step s
// (16 rows) from column chunk c0 (8 columns each) on.
__device__ __forceinline__ uint64_t operand_desc_t(uint32_t addr, int K, int s, int c0) {
    return smem_desc(addr + 128u * (uint32_t)c0 + 32u * (uint32_t)K * (uint32_t)s, 16u * (uint32_t)K, 128u);
}
// instruction descriptor with both operands read that way
__host__ __device__ constexpr uint32_t idesc_bf16_t(int M, int N) {
    return idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}

// D[tmem] (+)= A B^T for one 16-wide K step; issued by a single thread
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate));
}

// arrive on the mbarrier once every MMA this thread issued has completed
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// Wait for the phase with the given parity to complete, giving up after a
// bounded number of polls; returns false if it gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    const uint32_t a = smem_u32(bar);
    for (int i = 0; i < (1 << 20); ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// generic-proxy shared-memory writes -> visible to the tensor core (async proxy)
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Tensor-memory allocation (one full warp); the base address lands in *slot.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t base, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(ncols) : "memory");
}

// 16 consecutive FP32 columns of this thread's tensor-memory lane (warp-wide;
// warp w of a warpgroup reads lanes 32 (w % 4) .. 32 (w % 4) + 31)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 8 consecutive FP32 columns of this thread's tensor-memory lane, written;
// tmem_st_wait() before they are read back or the columns are used otherwise
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float* v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
                 "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

}  // namespace tc
}  // namespace vdw
