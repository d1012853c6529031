// npp_gemm.cu -- BF16 GEMM on the fifth-generation tensor cores.
//
// A persistent kernel: one CTA of 192 threads per SM walks 128 x BN tiles
// of C:
//   warp 0, one lane   TMA producer: K blocks of 64 (128 bytes of BF16, the
//                      128-byte swizzle atom) of A and B into a ring of
//                      STAGES shared-memory stages, completion counted by
//                      the stage's "full" mbarrier;
//   warp 1, one lane   MMA issuer: four tcgen05.mma (M = 128, N = BN,
//                      K = 16) per stage into one of two TMEM accumulators
//                      of BN FP32 columns (alternating by tile), then
//                      tcgen05.commit frees the stage ("empty"); after a
//                      tile's last stage a commit hands the accumulator to
//                      the epilogue ("tfull");
//   warps 2-5          epilogue: warp w reads TMEM lanes 32 (w % 4) ..
//                      32 (w % 4) + 31 (rows) with tcgen05.ld, stores them
//                      as FP32, and returns the accumulator
//                      ("tempty") -- while the MMAs of the next tile run on
//                      the other one.
// Every wait on an mbarrier is bounded (about a second of clock): on a
// timeout the CTA records an error code, stops issuing, waits (bounded) for
// the copies it issued, frees its TMEM and returns.
#include "npp_gemm.cuh"
#include "npp_tcgen05.cuh"

#include <cudaTypedefs.h>

#include <algorithm>

namespace npp {
namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int STAGES = 4;

template <int BN>
struct GemmShape {
    static constexpr int A_BYTES = BM * BK * 2;
    static constexpr int B_BYTES = BN * BK * 2;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024 + 128;   // + alignment slack + barriers
};

constexpr int GEMM_GROUP_M = 16;
constexpr int GEMM_THREADS = 192;

// one 128 x BN tile's accumulator rows (TMEM lanes 32 q .. 32 q + 31 at
// trow, this thread's row `row`) to global memory
template <int BN>
__device__ __forceinline__ void store_rows(float* C, int ldc, uint32_t trow, int row, int n0)
{
    const bool vec = (reinterpret_cast<uintptr_t>(C) & 31u) == 0;      // rows are whole 512-byte multiples
#pragma unroll 1
    for (int c = 0; c < BN; c += 16) {
        float v[16];
        tmem_ld16(trow + c, v);
        float* o = C + (size_t)row * ldc + n0 + c;
        if (vec) {
            store_32b(o, v);
            store_32b(o + 8, v + 8);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                reinterpret_cast<float4*>(o)[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
    }
}

// Tile `pid` in the grouped order: consecutive tiles walk GEMM_GROUP_M row
// tiles before the next column tile, so the CTAs busy at once share a few
// tiles of A and of B in L2.
__device__ __forceinline__ void unit_coords(int pid, int n_tiles, int m_tiles, int bn, int& m0, int& n0)
{
    const int per_group = GEMM_GROUP_M * n_tiles;
    const int first_m = (pid / per_group) * GEMM_GROUP_M;
    const int gsize = min(m_tiles - first_m, GEMM_GROUP_M);
    const int in_group = pid % per_group;
    m0 = (first_m + in_group % gsize) * BM;
    n0 = (in_group / gsize) * bn;
}

// Persistent GEMM: each CTA (one per SM) walks the work units
// blockIdx.x, blockIdx.x + gridDim.x, ...  The MMAs of a CTA's i-th unit go
// to TMEM accumulator i % 2 (BN columns each) while warps 2-5 drain the
// other one through the epilogue, so a tile's epilogue overlaps the next
// tile's MMAs; the operand ring and its barrier phases run on across units.
template <int BN>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
gemm_kernel(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, int M, int N, int K,
            float* C, int* err)
{
    using S = GemmShape<BN>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * S::STAGE_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* tfull = empty + STAGES;          // [2] accumulator ready for the epilogue
    uint64_t* tempty = tfull + 2;              // [2] accumulator drained by the epilogue (128 arrivals)
    uint64_t* done = tempty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    int* flags = reinterpret_cast<int*>(tmem_slot + 1);      // [0] abort, [1] issued, [2] consumed

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_tiles = N / BN, m_tiles = M / BM, units = n_tiles * m_tiles;
    const int nk = K / BK;                     // K blocks per unit

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], 128);
        }
        mbar_init(done, 1);
        flags[0] = 0;
        flags[1] = 0;
        flags[2] = 0;
        mbar_init_fence();
    }
    if (warp == 0) {
        __syncwarp();                          // after lane 0's set-up
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(2 * BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(tmem_slot);

    if (warp == 0 && lane == 0) {
        // TMA producer
        int g = 0;                             // K blocks issued by this CTA
        bool stop = false;
        for (int u = blockIdx.x; u < units && !stop; u += gridDim.x) {
            int m0, n0;
            unit_coords(u, n_tiles, m_tiles, BN, m0, n0);
            for (int kb = 0; kb < nk; ++kb, ++g) {
                const int s = g % STAGES;
                if (g >= STAGES && !mbar_wait(&empty[s], ((g / STAGES) - 1) & 1)) {
                    atomicExch(&flags[0], 1);
                    stop = true;
                    break;
                }
                if (*reinterpret_cast<volatile int*>(&flags[0])) {
                    stop = true;
                    break;
                }
                uint8_t* st = smem + s * S::STAGE_BYTES;
                const int kc = kb * BK;
                mbar_expect_tx(&full[s], S::STAGE_BYTES);
                tma_load_2d(st, &ta, kc, m0, &full[s]);
                tma_load_2d(st + S::A_BYTES, &tb, kc, n0, &full[s]);
            }
        }
        flags[1] = g;
    } else if (warp == 1 && lane == 0) {
        // MMA issuer
        constexpr uint32_t idesc = mma_idesc(BN);
        int g = 0, i = 0;
        bool stop = false;
        for (int u = blockIdx.x; u < units && !stop; u += gridDim.x, ++i) {
            const int b = i & 1;
            // the accumulator's previous tile drained (its first use passes at once)
            if (!mbar_wait(&tempty[b], ((i >> 1) & 1) ^ 1)) {
                atomicExch(&flags[0], 1);
                break;
            }
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)(b * BN);
            for (int kb = 0; kb < nk; ++kb, ++g) {
                const int s = g % STAGES;
                if (!mbar_wait(&full[s], (g / STAGES) & 1)) {
                    atomicExch(&flags[0], 1);
                    stop = true;
                    break;
                }
                tc_fence_after();
                const uint32_t a0 = smem_u32(smem + s * S::STAGE_BYTES);
                const uint32_t b0 = a0 + S::A_BYTES;
#pragma unroll
                for (int j = 0; j < BK / 16; ++j)
                    mma_bf16(acc, sw128_desc(a0 + j * 32), sw128_desc(b0 + j * 32), idesc, (kb | j) != 0);
                mma_commit(&empty[s]);
            }
            if (!stop) mma_commit(&tfull[b]);  // arrives once this unit's MMAs have completed
        }
        flags[2] = g;
        mma_commit(done);
    } else if (warp >= 2) {
        // epilogue: warp w reads TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31
        const int q = warp & 3;
        int i = 0;
        for (int u = blockIdx.x; u < units; u += gridDim.x, ++i) {
            const int b = i & 1;
            const bool ok = mbar_wait(&tfull[b], (i >> 1) & 1);
            // (one answer for the warp, whose lanes the vote brings together:
            // the accumulator reads are the whole warp's)
            if (!__all_sync(0xffffffffu, ok && !*reinterpret_cast<volatile int*>(&flags[0]))) {
                atomicExch(&flags[0], 1);
                break;
            }
            tc_fence_after();
            int m0, n0;
            unit_coords(u, n_tiles, m_tiles, BN, m0, n0);
            store_rows<BN>(C, N, tmem + (uint32_t)(b * BN) + ((uint32_t)(q * 32) << 16), m0 + q * 32 + lane, n0);
            tc_fence_before();
            mbar_arrive(&tempty[b]);
        }
    }
    __syncwarp();
    __syncthreads();
    if (threadIdx.x == 0) {
        // every MMA complete before the TMEM goes back; after a timeout the
        // copies issued but never consumed land first (bounded waits)
        const bool ok = mbar_wait(done, 0);
        if (!ok || *reinterpret_cast<volatile int*>(&flags[0])) {
            if (err) atomicExch(err, 1);
            for (int g = flags[2]; g < flags[1]; ++g) mbar_wait(&full[g % STAGES], (g / STAGES) & 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
    }
}

// The same GEMM on CTA pairs (cta_group::2): a pair takes 256 x 256 tiles;
// each CTA loads its 128 rows of A and its 128 of the tile's 256 rows of B,
// so a stage is 32 KB instead of 48 (six stages in flight instead of four)
// and every byte of B is read into one SM's shared memory instead of two.
// The even CTA's MMA lane issues for both; copies of both CTAs count on its
// "full" barriers, its commits free the stage and hand the accumulator over
// in both, and both epilogues return it on its "tempty" barriers.
// M = N = K = 8192 on GB300: 612 us under the profiler (1797 TFLOP/s; the
// 128 x 256 tiles of one CTA take 710), 710 us against 756 in back-to-back
// calls, where the power limit holds both. Grouping 8 or 4 row tiles instead
// of 16: 711 and 730 us against 720, within what runs differ by.
constexpr int PAIR_STAGES = 6;
constexpr int PAIR_STAGE = 2 * BM * BK * 2;
constexpr int PAIR_SMEM = PAIR_STAGES * PAIR_STAGE + 1024 + 256;

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GEMM_THREADS, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, int M, int N, int K,
                 float* C, int* err)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + PAIR_STAGES * PAIR_STAGE);
    uint64_t* empty = full + PAIR_STAGES;
    uint64_t* tfull = empty + PAIR_STAGES;
    uint64_t* tempty = tfull + 2;              // both CTAs' 128 epilogue threads
    uint64_t* done = tempty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    int* flags = reinterpret_cast<int*>(tmem_slot + 1);      // [0] abort, [1] issued, [2] consumed

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int n_tiles = N / 256, m_tiles = M / 256, units = n_tiles * m_tiles, nk = K / BK;
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < PAIR_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], 256);
        }
        mbar_init(done, 1);
        flags[0] = flags[1] = flags[2] = 0;
        mbar_init_fence();
    }
    if (warp == 0) {
        __syncwarp();                          // after lane 0's set-up
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();                            // the peer's barriers are ready
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(tmem_slot);

    if (warp == 0 && lane == 0) {
        // TMA producer of this CTA's halves
        int g = 0;
        bool stop = false;
        for (int u = pair; u < units && !stop; u += pairs) {
            int m0, n0;
            unit_coords(u, n_tiles, m_tiles, 256, m0, n0);
            m0 = 2 * m0 + 128 * (int)rank;     // unit_coords counts row tiles of 128
            n0 += 128 * (int)rank;
            for (int kb = 0; kb < nk; ++kb, ++g) {
                const int s = g % PAIR_STAGES;
                if (g >= PAIR_STAGES && !mbar_wait_cluster(&empty[s], ((g / PAIR_STAGES) - 1) & 1))
                    atomicExch(&flags[0], 1);
                if (*reinterpret_cast<volatile int*>(&flags[0])) {
                    stop = true;
                    break;
                }
                uint8_t* st = smem + s * PAIR_STAGE;
                if (rank == 0) mbar_expect_tx(&full[s], 2 * PAIR_STAGE);
                const uint32_t bar = leader_addr(&full[s]);
                tma_load_2d_pair(st, &ta, kb * BK, m0, bar);
                tma_load_2d_pair(st + PAIR_STAGE / 2, &tb, kb * BK, n0, bar);
            }
        }
        flags[1] = g;
    } else if (warp == 1 && lane == 0 && rank == 0) {
        constexpr uint32_t idesc = mma_idesc(256, false, false, 256);
        int g = 0, i = 0;
        bool stop = false;
        for (int u = pair; u < units && !stop; u += pairs, ++i) {
            const int b = i & 1;
            if (!mbar_wait_cluster(&tempty[b], ((i >> 1) & 1) ^ 1)) {
                atomicExch(&flags[0], 1);
                break;
            }
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)(b * 256);
            for (int kb = 0; kb < nk; ++kb, ++g) {
                const int s = g % PAIR_STAGES;
                if (!mbar_wait_cluster(&full[s], (g / PAIR_STAGES) & 1)) {
                    atomicExch(&flags[0], 1);
                    stop = true;
                    break;
                }
                tc_fence_after();
                const uint32_t a0 = smem_u32(smem + s * PAIR_STAGE), b0 = a0 + PAIR_STAGE / 2;
#pragma unroll
                for (int j = 0; j < BK / 16; ++j)
                    mma_bf16_pair(acc, sw128_desc(a0 + j * 32), sw128_desc(b0 + j * 32), idesc, (kb | j) != 0);
                mma_commit_pair(&empty[s]);
            }
            if (!stop) mma_commit_pair(&tfull[b]);
        }
        flags[2] = g;
        mma_commit_pair(done);
    } else if (warp >= 2) {
        const int q = warp & 3;
        int i = 0;
        for (int u = pair; u < units; u += pairs, ++i) {
            const int b = i & 1;
            const bool ok = mbar_wait_cluster(&tfull[b], (i >> 1) & 1);
            // (one answer for the warp, whose lanes the vote brings together:
            // the accumulator reads are the whole warp's)
            if (!__all_sync(0xffffffffu, ok && !*reinterpret_cast<volatile int*>(&flags[0]))) {
                atomicExch(&flags[0], 1);
                break;
            }
            tc_fence_after();
            int m0, n0;
            unit_coords(u, n_tiles, m_tiles, 256, m0, n0);
            store_rows<256>(C, N, tmem + (uint32_t)(b * 256) + ((uint32_t)(q * 32) << 16),
                            2 * m0 + 128 * (int)rank + q * 32 + lane, n0);
            tc_fence_before();
            arrive_cluster(leader_addr(&tempty[b]));
        }
    }
    __syncwarp();
    __syncthreads();
    if (threadIdx.x == 0) {
        // every MMA complete before the TMEM goes back; after a timeout the
        // copies issued but never consumed land first (bounded waits)
        const bool ok = mbar_wait_cluster(done, 0);
        if (!ok || *reinterpret_cast<volatile int*>(&flags[0])) {
            if (err) atomicExch(err, 1);
            if (rank == 0)
                for (int g = flags[2]; g < flags[1]; ++g) mbar_wait_cluster(&full[g % PAIR_STAGES], (g / PAIR_STAGES) & 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();                            // neither CTA leaves while the other uses its memory
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

int sm_count()
{
    static int cnt[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 148;
    if (cnt[dev] == 0) {
        int c = 0;
        if (cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || c <= 0) c = 148;
        cnt[dev] = c;
    }
    return cnt[dev];
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

}  // namespace

cudaError_t make_tmap_bf16(CUtensorMap* map, const void* base, int rows, int cols, int box_rows)
{
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    if ((reinterpret_cast<uintptr_t>(base) & 15u) || cols % 64 || rows % box_rows) return cudaErrorInvalidValue;
    cuuint64_t dims[2] = { (cuuint64_t)cols, (cuuint64_t)rows };
    cuuint64_t strides[1] = { (cuuint64_t)cols * 2 };
    cuuint32_t box[2] = { 64u, (cuuint32_t)box_rows };
    cuuint32_t estr[2] = { 1u, 1u };
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Whether the pair kernel takes the product: whole 256 x 256 tiles, and
// enough of them to give every pair of SMs one (fewer tiles fill more SMs as
// 128-row tiles).
bool gemm_pairs(int M, int N)
{
    return M % 256 == 0 && N % 256 == 0 && (M / 256) * (N / 256) >= sm_count() / 2;
}

cudaError_t launch_gemm(const CUtensorMap& ta, const CUtensorMap& tb, int M, int N, int K, int bn, int box_b, float* C,
                        int* err, cudaStream_t s)
{
    if (M % BM || K % BK || K < BK || (bn != 128 && bn != 256) || N % bn) return cudaErrorInvalidValue;
    if (bn == 256 && box_b == 128) {
        cudaError_t e = cudaFuncSetAttribute(gemm_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PAIR_SMEM);
        if (e != cudaSuccess) return e;
        const int pairs = std::min((M / 256) * (N / 256), sm_count() / 2);
        gemm_pair_kernel<<<2 * pairs, GEMM_THREADS, PAIR_SMEM, s>>>(ta, tb, M, N, K, C, err);
        return cudaGetLastError();
    }
    const int grid = std::min((M / BM) * (N / bn), sm_count());
    if (bn == 256) {
        const int smem = GemmShape<256>::SMEM;
        cudaError_t e = cudaFuncSetAttribute(gemm_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        gemm_kernel<256><<<grid, GEMM_THREADS, smem, s>>>(ta, tb, M, N, K, C, err);
    } else {
        const int smem = GemmShape<128>::SMEM;
        cudaError_t e = cudaFuncSetAttribute(gemm_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        gemm_kernel<128><<<grid, GEMM_THREADS, smem, s>>>(ta, tb, M, N, K, C, err);
    }
    return cudaGetLastError();
}

}  // namespace npp
