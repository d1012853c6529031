// npp_tmem.cuh -- tensor memory (256 KB per SM: 128 lanes x 512 columns of 32
// bits) as plain per-warp storage, as inline PTX.  A warp reaches the 32
// lanes of its quarter (warp index modulo 4); one column is one 32-bit value
// per thread.  Every instruction here but the fences is the whole warp's
// (.sync.aligned): after code that parts its lanes, callers __syncwarp first.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

#include "npp_async.cuh"

namespace npp {

// A block's TMEM columns (a power of two, 32 or more), allocated by its
// first warp and handed to all; every thread of the block calls both.  The
// allocation waits in hardware while other resident blocks hold the columns
// it needs; a block holds one allocation only, so the others always end.
template <int COLS>
__device__ __forceinline__ uint32_t tmem_alloc(uint32_t* slot)
{
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(slot)), "n"(COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return *reinterpret_cast<volatile uint32_t*>(slot);
}

template <int COLS>
__device__ __forceinline__ void tmem_free(uint32_t tmem)
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(COLS) : "memory");
}

// Sixteen consecutive columns of a lane.
struct Tmem16 {
    uint32_t r[16];
    __device__ __forceinline__ float f(int i) const { return __uint_as_float(r[i]); }
    __device__ __forceinline__ unsigned long long pair(int i) const
    {
        unsigned long long d;
        asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(r[2 * i]), "r"(r[2 * i + 1]));
        return d;
    }
};

// columns taddr .. taddr + 15 of this warp's 32 lanes, valid after
// tmem_wait_ld (which waits for every read the warp has issued)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, Tmem16& v)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v.r[0]), "=r"(v.r[1]), "=r"(v.r[2]), "=r"(v.r[3]), "=r"(v.r[4]), "=r"(v.r[5]), "=r"(v.r[6]),
          "=r"(v.r[7]), "=r"(v.r[8]), "=r"(v.r[9]), "=r"(v.r[10]), "=r"(v.r[11]), "=r"(v.r[12]), "=r"(v.r[13]),
          "=r"(v.r[14]), "=r"(v.r[15])
        : "r"(taddr));
}

// the registers pass through the wait, so that no use of them moves before it
__device__ __forceinline__ void tmem_wait_ld(Tmem16& v)
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
        : "+r"(v.r[0]), "+r"(v.r[1]), "+r"(v.r[2]), "+r"(v.r[3]), "+r"(v.r[4]), "+r"(v.r[5]), "+r"(v.r[6]),
          "+r"(v.r[7]), "+r"(v.r[8]), "+r"(v.r[9]), "+r"(v.r[10]), "+r"(v.r[11]), "+r"(v.r[12]), "+r"(v.r[13]),
          "+r"(v.r[14]), "+r"(v.r[15])
        :: "memory");
}

__device__ __forceinline__ void tmem_st4(uint32_t taddr, const float4& v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                 ::"r"(taddr), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)),
                 "r"(__float_as_uint(v.w)) : "memory");
}

__device__ __forceinline__ void tmem_st2(uint32_t taddr, const float2& v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};"
                 ::"r"(taddr), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)) : "memory");
}

__device__ __forceinline__ void tmem_wait_st()
{
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

}  // namespace npp
