// tc5.cuh -- tcgen05 (5th-generation tensor core) device helpers shared by the GEMM and
// convolution kernels (PTX ISA, "Tensor Core 5th Generation Family Instructions").
#pragma once
#include "tma.cuh"

namespace mgmc {
namespace tc5 {

// shared-memory matrix descriptor: start address >> 4 (bits 0-13), leading byte offset >> 4
// (16-29), stride byte offset >> 4 (32-45), descriptor version 1 (46-47), swizzle mode
// (61-63: 2 = 128 B, 4 = 64 B, 6 = 32 B)
__device__ __forceinline__ unsigned long long desc(unsigned saddr, unsigned lbo, unsigned sbo, unsigned swizzle)
{
    return (unsigned long long)((saddr & 0x3FFFFu) >> 4) | ((unsigned long long)(lbo >> 4) << 16) |
           ((unsigned long long)(sbo >> 4) << 32) | (1ull << 46) | ((unsigned long long)swizzle << 61);
}
// swizzle mode of rows of `bytes` bytes
__host__ __device__ constexpr unsigned swizzle_of(int bytes) { return bytes == 128 ? 2u : bytes == 64 ? 4u : 6u; }

// instruction descriptor of kind::f16: D = F32, A = B = BF16, M = 128; `mn`: both operands
// MN-major (bits 15, 16)
__device__ __forceinline__ unsigned idesc(int n, bool mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (1u << 15) | (1u << 16) : 0u) | ((unsigned)(n >> 3) << 17) |
           ((unsigned)(128 >> 4) << 24);
}
__device__ __forceinline__ void mma(unsigned tmem_d, unsigned long long da, unsigned long long db, unsigned id,
                                    unsigned accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(id), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void commit(unsigned long long* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_addr(bar))
                 : "memory");
}
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void alloc(unsigned* slot, unsigned cols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(slot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void dealloc(unsigned base, unsigned cols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(base), "r"(cols) : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns of TMEM into r[0..31] (this warp's lanes)
__device__ __forceinline__ void ld32(unsigned taddr, unsigned* r)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void arrive(unsigned long long* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c, int x, int y, int b,
                                            unsigned long long* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];\n" ::"r"(smem_addr(dst)),
        "l"(map), "r"(c), "r"(x), "r"(y), "r"(b), "r"(smem_addr(bar))
        : "memory");
}

// Bound of the producer's and the epilogue's waits, from a kernel's wait_ns (see mbar_wait).  The MMA
// issuer's waits, one a chunk on the critical path, have the default bound as a constant (a bound
// held in registers cost a product of 36 chunks 1.4 of 17 us); with a negative wait_ns it gives up
// before its first operands, so that the others are caught waiting
__device__ __forceinline__ long long role_limit(long long wait_ns) { return wait_ns < 0 ? -wait_ns : wait_ns; }

// position in a ring of n slots: slot and the parity of its current use (32-bit counters: a
// 64-bit remainder per chunk cost the issuing thread more than the chunk's MMAs)
struct RingPos {
    int slot = 0;
    unsigned par = 0;
    __device__ __forceinline__ void next(int n)
    {
        if (++slot == n) {
            slot = 0;
            par ^= 1u;
        }
    }
    __device__ __forceinline__ int ahead(int d, int n) const { return slot + d >= n ? slot + d - n : slot + d; }
};

}  // namespace tc5
}  // namespace mgmc
