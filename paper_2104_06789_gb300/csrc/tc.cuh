// Fifth-generation tensor core (tcgen05), bulk-copy and mbarrier helpers shared
// by the kernels that issue them: inline PTX only, no state.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace vd {

__device__ __forceinline__ uint32_t smem_addr(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void tc_mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ bool tc_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred P;\n mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n selp.u32 %0, 1, 0, P;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}

__device__ __forceinline__ void tc_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Shared-memory matrix descriptor, K-major without swizzle: start, leading
// (K-direction core-matrix) offset, stride (M/N-direction 8-row group) offset.
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// MMAs, commits, copies and expected bytes are issued by one elected lane of a converged
// warp, which keeps descriptors and barriers in uniform registers; the same loop inside
// an `if (lane == 0)` moves each operand over instruction by instruction: three waits,
// four MMAs (M = 128, N = 96) and two commits took 493 cycles a round there and take
// 283 here, 226 of them the MMAs' shared-memory reads.
__device__ __forceinline__ void tc_mma_elect(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile("{\n .reg .pred p, q;\n elect.sync _|q, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
                 " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void tc_commit_elect(uint32_t bar)
{
    asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n"
                 " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_expect_tx_elect(uint32_t bar, uint32_t bytes)
{
    asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n"
                 " @q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}" ::"r"(bar), "r"(bytes) : "memory");
}

// Contiguous global -> shared copy (16-byte aligned, a multiple of 16 bytes)
// completing on an mbarrier.
__device__ __forceinline__ void tc_bulk_g2s_elect(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n"
                 " @q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n}"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// Keeps what reads columns loaded from tensor memory behind the wait for them.
template <int NC>
__device__ __forceinline__ void tc_hold(uint32_t* r)
{
#pragma unroll
    for (int i = 0; i < NC; ++i) asm volatile("" : "+r"(r[i]));
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

}  // namespace vd
