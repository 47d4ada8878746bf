// pond_tc.cuh -- 5th-generation tensor-core primitives (tcgen05, TMEM) for sm_103a.
//
// Operands live in shared memory as BF16 in the K-major layout without swizzle: the tile
// is cut into 8-row x 8-element "core matrices" of 128 contiguous bytes (8 rows of 16 B);
// core matrices adjacent along K are LBO = 128 B apart and 8-row groups are
// SBO = (K/8) * 128 B apart.  One tcgen05.mma (kind::f16, K = 16) consumes two core
// matrices along K, so successive K steps advance the descriptors by 256 B.  Accumulators
// are FP32 in tensor memory: an M = 128 tile occupies lanes 0..127, row i in lane i; warp w
// of the CTA reads lanes 32 (w % 4) .. 32 (w % 4) + 31.
//
// Every wait on an mbarrier is bounded; on time-out the caller records an error, releases
// its tensor memory and returns.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace pond {
namespace tc {

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// byte offset of element (r, k) of a K-major, unswizzled BF16 operand with K columns
__host__ __device__ constexpr uint32_t kmajor_offset(uint32_t r, uint32_t k, uint32_t K)
{
    return (r >> 3) * (K / 8) * 128u + (k >> 3) * 128u + (r & 7u) * 16u + (k & 7u) * 2u;
}

// shared-memory matrix descriptor: start address, leading (K) and stride (8-row) byte
// offsets, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return uint64_t((saddr >> 4) & 0x3FFFu) | (uint64_t((lbo >> 4) & 0x3FFFu) << 16) |
           (uint64_t((sbo >> 4) & 0x3FFFu) << 32) | (uint64_t(1) << 46);
}

// instruction descriptor of kind::f16: D FP32, A and B BF16, M x N, both K-major or (mn) both
// MN-major
__host__ __device__ constexpr uint32_t idesc_bf16(uint32_t M, uint32_t N, bool mn = false)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? 3u << 15 : 0u) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void commit(uint64_t *mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(mbar)) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *mbar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(mbar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// bounded wait for the given phase parity; false on time-out
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t parity, long long max_polls)
{
    const uint32_t a = smem_addr(mbar);
    for (long long i = 0; i < max_polls; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// smem written by ordinary stores, about to be read by the tensor core (async proxy)
__device__ __forceinline__ void fence_smem_to_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// tensor-memory allocation by one full warp; the base address lands in *dst (shared)
__device__ __forceinline__ void tmem_alloc(uint32_t *dst, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(dst)), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t base, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(ncols) : "memory");
}

// 16 consecutive FP32 columns of this thread's lane (warp-collective)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 64 consecutive FP32 columns of this thread's lane, load and wait in one statement so no
// use of the registers can be scheduled before the wait (warp-collective)
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float *v)
{
    uint32_t r[64];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 {"
        "%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15,"
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31,"
        "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47,"
        "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
          "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
          "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]),
          "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
          "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}

// D[128 x N] = A[128 x K] B[N x K]^T; issued by one thread; A, B K-major in shared memory, stored
// with Ka and Kb columns
__device__ __forceinline__ void gemm_issue(uint32_t d_tmem, const void *A, uint32_t Ka, const void *B, uint32_t Kb, uint32_t K,
                                           uint32_t N)
{
    const uint32_t id = idesc_bf16(128, N);
    const uint32_t a0 = smem_addr(A), b0 = smem_addr(B);
    for (uint32_t ks = 0; ks < K / 16; ++ks) {
        const uint64_t ad = smem_desc(a0 + ks * 256u, 128u, (Ka / 8) * 128u);
        const uint64_t bd = smem_desc(b0 + ks * 256u, 128u, (Kb / 8) * 128u);
        mma_bf16(d_tmem, ad, bd, id, ks > 0 ? 1u : 0u);
    }
}

// D[128 x N] (+)= A^T B over K rows of A [K][Ca] and B [K][Cb], stored as for gemm_issue: read
// MN-major, core matrices are 128 B apart along the units (stride offset) and a row group's
// (C/8) * 128 B apart along K (leading offset).  Units of A past Ca give rows of D that mean nothing.
__device__ __forceinline__ void gemm_issue_mn(uint32_t d_tmem, const void *A, uint32_t Ca, const void *B, uint32_t Cb, uint32_t K,
                                              uint32_t N, bool accumulate)
{
    const uint32_t id = idesc_bf16(128, N, true);
    const uint32_t a0 = smem_addr(A), b0 = smem_addr(B), la = (Ca / 8) * 128u, lb = (Cb / 8) * 128u;
    for (uint32_t ks = 0; ks < K / 16; ++ks) {
        const uint64_t ad = smem_desc(a0 + ks * 2u * la, la, 128u);
        const uint64_t bd = smem_desc(b0 + ks * 2u * lb, lb, 128u);
        mma_bf16(d_tmem, ad, bd, id, (accumulate || ks > 0) ? 1u : 0u);
    }
}

}  // namespace tc
}  // namespace pond
