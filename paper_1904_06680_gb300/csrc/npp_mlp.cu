// npp_mlp.cu -- the sampling-proposal network on the fifth-generation tensor
// cores: one kernel for the whole forward pass (with the outputs' mean and
// std, or the loss and its gradient), one for the activations' gradients and
// one for the three weight gradients.
//
// Why fused: a layer's product at these sizes takes a few microseconds of
// tensor-core time, less than a launch, the pipeline's fill and the trip of
// its activations through memory.  A CTA takes 128 batch rows through all
// layers; between layers the activations go from tensor memory through the
// bias and ReLU straight into shared memory as the next product's operand
// (BF16, K-major, 128-byte swizzle).  The weight gradients read the
// activations row-major as they are (MN-major operands), so nothing is
// stored transposed.  Measured on GB300: training step at batch 8192 (all
// launches) 187 -> 84 us; a forward pass of 300 rows with the encoding of
// their scenes 61 -> 28 us.
//
// In a training step each kernel starts while the one before it runs
// (programmatic dependent launch), on the SMs that one leaves idle: the
// backward pass fills 64 of 152 at batch 8192, and dW3 needs nothing of it.
// A kernel lets the next one start only after its own wait, so what lies two
// launches back is complete; see the waits.  16 steps and two reads of the
// parameters so 1638 -> 1436 us.
//
// Every CTA: one TMA producer lane, one MMA-issuing lane, eight epilogue
// warps (two per TMEM lane quarter, each half of the columns).  All waits
// are bounded; on a timeout the CTA records an error, stops issuing, waits
// (bounded) for its copies, frees its TMEM and returns.
#include "npp_launch.cuh"
#include "npp_mlp.cuh"
#include "npp_tcgen05.cuh"

#include <algorithm>

namespace npp {
namespace {

typedef __nv_bfloat16 bf16;

constexpr int THREADS = 320;               // producer, MMA issuer, 8 epilogue warps
constexpr int EPI_THREADS = 256;
constexpr int TILE_M = 128;
constexpr int A_BLOCK = TILE_M * 128;      // an operand block: 128 rows x 64 BF16 of K
constexpr int W_BLOCK = 256 * 128;         // a weight block: 256 x 64 BF16

// barriers and flags of a CTA
template <int STAGES>
struct Pipe {
    uint64_t full[STAGES], empty[STAGES];
    uint64_t tfull[2];                     // accumulator ready for the epilogue
    uint64_t tempty[2];                    // accumulator drained (EPI_THREADS arrivals)
    uint64_t aready;                       // operand written by the epilogue warps
    uint64_t done;
    uint32_t tmem;
    int flags[3];                          // [0] abort, [1] blocks issued, [2] blocks consumed
};

template <int STAGES>
__device__ __forceinline__ uint32_t pipe_init(Pipe<STAGES>& p)
{
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&p.full[s], 1);
            mbar_init(&p.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&p.tfull[b], 1);
            mbar_init(&p.tempty[b], EPI_THREADS);
        }
        mbar_init(&p.aready, EPI_THREADS);
        mbar_init(&p.done, 1);
        p.flags[0] = p.flags[1] = p.flags[2] = 0;
        mbar_init_fence();
    }
    if (warp == 0) {
        __syncwarp();                          // after lane 0's set-up
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&p.tmem)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    return *reinterpret_cast<volatile uint32_t*>(&p.tmem);
}

template <int STAGES>
__device__ __forceinline__ bool aborted(Pipe<STAGES>& p) { return *reinterpret_cast<volatile int*>(&p.flags[0]) != 0; }

template <int STAGES>
__device__ __forceinline__ void pipe_end(Pipe<STAGES>& p, uint32_t tmem, int* err)
{
    __syncwarp();
    __syncthreads();
    if (threadIdx.x == 0) {
        // every MMA complete before the TMEM goes back; after a timeout the
        // copies issued but never consumed land first (bounded waits)
        const bool ok = mbar_wait(&p.done, 0);
        if (!ok || aborted(p)) {
            if (err) atomicExch(err, 1);
            for (int g = p.flags[2]; g < p.flags[1]; ++g) mbar_wait(&p.full[g % STAGES], (g / STAGES) & 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// Epilogue side, after a wait: whether every lane's was in time and nothing
// aborted, the same answer for the whole warp.  The vote also brings its lanes
// together: the accumulator reads that follow are the whole warp's.
template <int STAGES>
__device__ __forceinline__ bool epilogue_go(Pipe<STAGES>& p, bool ok) { return __all_sync(0xffffffffu, ok && !aborted(p)); }

// Producer side: the next stage, free; false to stop.
template <int STAGES>
__device__ __forceinline__ bool stage_free(Pipe<STAGES>& p, int g)
{
    const int s = g % STAGES;
    if (g >= STAGES && !mbar_wait(&p.empty[s], ((g / STAGES) - 1) & 1)) atomicExch(&p.flags[0], 1);
    return !aborted(p);
}

// address of 16-byte chunk c16 (0..7) of row r in a K-major 128-byte-swizzled
// block of 128-byte rows
__device__ __forceinline__ uint32_t sw_off(int r, int c16) { return (uint32_t)(r * 128 + ((c16 ^ (r & 7)) << 4)); }

// sixteen consecutive K columns k0 (a multiple of 16) of row r of a K-major
// operand stored in blocks of 64 columns
__device__ __forceinline__ void put_row16(uint8_t* A, int r, int k0, const bf16* v)
{
    uint8_t* blk = A + (k0 >> 6) * A_BLOCK;
    const uint4* s = reinterpret_cast<const uint4*>(v);
    const int c = (k0 & 63) >> 3;
    *reinterpret_cast<uint4*>(blk + sw_off(r, c)) = s[0];
    *reinterpret_cast<uint4*>(blk + sw_off(r, c + 1)) = s[1];
}

// sixteen bias values (16-byte aligned)
__device__ __forceinline__ void load16(const float* p, float* v)
{
    const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 t = q[i];
        v[4 * i] = t.x; v[4 * i + 1] = t.y; v[4 * i + 2] = t.z; v[4 * i + 3] = t.w;
    }
}

// ------------------------------------------------------------------ forward
constexpr int FW_STAGES = 3;
constexpr int FW_BIAS = 2 * MLP_HID + MLP_D3;              // b1, b2, the means' and the log-stds' biases
constexpr int FW_SCRATCH = 32 * 34 * 4 + 256;              // per epilogue warp (see Scratch), 4608 bytes
constexpr int FW_SMEM = 4 * A_BLOCK + FW_STAGES * W_BLOCK + 1024 + 4 * FW_BIAS + 8 * FW_SCRATCH +
                        (int)sizeof(Pipe<FW_STAGES>);
constexpr int FW_K1 = 80;                  // layer 1's K: 72 inputs and 8 zeros

// A warp's scratch turns row-per-lane registers (the accumulator's layout)
// into row-wise global accesses and back: 32 rows x 32 columns, FP32 rows 34
// words apart, BF16 rows 18 (64-bit accesses row per lane and 32-bit ones
// along the rows hit different banks).  Without it every lane's access would
// touch a line of its own (rows are 1800 or 2048 bytes apart).
constexpr int SC_F32 = 34, SC_BF16 = 18;

// rows m0 .. m0 + 31, columns i0 .. i0 + 31 of an [n][450] FP32 matrix: lane l
// reads columns 2 (l % 16), + 1 of rows l / 16 + 2 k; zero beyond row n and
// column 449 (i0 even, 450 even: a pair is inside or outside)
__device__ __forceinline__ void fetch_rows(const float* p, bool vec, int m0, int n, int i0, int lane, float2 (&v)[16])
{
    const int c = i0 + 2 * (lane & 15);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int row = m0 + 2 * k + (lane >> 4);
        v[k] = make_float2(0.f, 0.f);
        if (row < n && c < MLP_NTH) {
            const float* q = p + (size_t)row * MLP_NTH + c;
            if (vec) v[k] = __ldg(reinterpret_cast<const float2*>(q));
            else v[k] = make_float2(q[0], q[1]);
        }
    }
}
__device__ __forceinline__ void rows_to_scratch(float* sc, int lane, const float2 (&v)[16])
{
#pragma unroll
    for (int k = 0; k < 16; ++k)
        *reinterpret_cast<float2*>(sc + (2 * k + (lane >> 4)) * SC_F32 + 2 * (lane & 15)) = v[k];
}
// the scratch's FP32 rows to columns i0 .. of an [n][450] matrix
__device__ __forceinline__ void scratch_to_rows(const float* sc, float* p, bool vec, int m0, int n, int i0, int lane)
{
    const int c = i0 + 2 * (lane & 15);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int row = m0 + 2 * k + (lane >> 4);
        if (row < n && c < MLP_NTH) {
            const float2 t = *reinterpret_cast<const float2*>(sc + (2 * k + (lane >> 4)) * SC_F32 + 2 * (lane & 15));
            float* q = p + (size_t)row * MLP_NTH + c;
            if (vec) {
                *reinterpret_cast<float2*>(q) = t;
            } else {
                q[0] = t.x;
                q[1] = t.y;
            }
        }
    }
}

// A unit is a row tile and a group of its output tiles; a CTA walks units
// blockIdx.x, + gridDim.x, ...  Per unit the products are layer 1 (K = 80),
// layer 2 and one output tile after the other, each 128 x 256 in one of the
// two TMEM accumulators by turns: an output tile's epilogue runs while the
// next tile's MMAs fill the other one.
template <bool TRAIN>
__global__ void __launch_bounds__(THREADS, 1)
mlp_forward_kernel(const __grid_constant__ MlpForwardMaps maps, const MlpForward f)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* A = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* ring = A + 4 * A_BLOCK;
    // biases: b1 [256], b2 [256], means [512], log-stds [512] (zero beyond 449)
    float* bias = reinterpret_cast<float*>(ring + FW_STAGES * W_BLOCK);
    uint8_t* scratch = reinterpret_cast<uint8_t*>(bias + FW_BIAS);
    Pipe<FW_STAGES>& p = *reinterpret_cast<Pipe<FW_STAGES>*>(scratch + 8 * FW_SCRATCH);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < FW_BIAS; i += THREADS) {
        const int o = i < 2 * MLP_HID ? 0 : (i - 2 * MLP_HID) % (MLP_D3 / 2);
        bias[i] = i < MLP_HID ? f.b1[i] : i < 2 * MLP_HID ? f.b2[i - MLP_HID]
                : o >= MLP_NTH ? 0.0f : f.b3[i < 2 * MLP_HID + MLP_D3 / 2 ? o : MLP_NTH + o];
    }
    const uint32_t tmem = pipe_init(p);        // a block barrier: the biases are in
    start_next();
    const int tiles = (f.n + TILE_M - 1) / TILE_M, units = tiles * f.groups, tpu = 4 / f.groups;

    if (warp == 0 && lane == 0) {
        // producer: W1's 2 K blocks, W2's 4, then 4 per output tile
        int g = 0;
        bool go = true;
        for (int u = blockIdx.x; u < units && go; u += gridDim.x) {
            const int t0 = (u % f.groups) * tpu;
            for (int k = 0; k < 6 + 4 * tpu; ++k) {
                if (!(go = stage_free(p, g))) break;
                const int s = g % FW_STAGES;
                mbar_expect_tx(&p.full[s], W_BLOCK);
                uint8_t* st = ring + s * W_BLOCK;
                if (k < 2) tma_load_2d(st, &maps.w1, k * 64, 0, &p.full[s]);
                else if (k < 6) tma_load_2d(st, &maps.w2, (k - 2) * 64, 0, &p.full[s]);
                else tma_load_2d(st, &maps.w3, ((k - 6) & 3) * 64, (t0 + ((k - 6) >> 2)) * 256, &p.full[s]);
                ++g;
            }
        }
        p.flags[1] = g;
    } else if (warp == 1 && lane == 0) {
        // MMA issuer; it also stores the hidden activations, which lie in
        // shared memory as operands, for the backward pass
        constexpr uint32_t idesc = mma_idesc(256);
        int g = 0, layer = 0, ready = 0;
        bool go = true;
        for (int u = blockIdx.x; u < units && go; u += gridDim.x) {
            const bool store = TRAIN && u % f.groups == 0;  // one unit of a row tile stores
            for (int l = 0; l < 2 + tpu && go; ++l, ++layer) {
                const int b = layer & 1;
                bool ok = mbar_wait(&p.tempty[b], ((layer >> 1) & 1) ^ 1);
                if (l < 3) ok = ok && mbar_wait(&p.aready, ready++ & 1);     // a new operand (output tiles share one)
                if (!ok || aborted(p)) { atomicExch(&p.flags[0], 1); go = false; break; }
                tc_fence_after();
                const bool st = store && (l == 1 || l == 2);
                if (st) {
                    for (int kb = 0; kb < 4; ++kb)
                        tma_store_2d(l == 1 ? &maps.h1 : &maps.h2, A + kb * A_BLOCK, kb * 64, u / f.groups * TILE_M);
                    bulk_store_commit();
                }
                const uint32_t acc = tmem + (uint32_t)(b * 256);
                const int nk = l == 0 ? 2 : 4;
                for (int kb = 0; kb < nk; ++kb, ++g) {
                    const int s = g % FW_STAGES;
                    if (!mbar_wait(&p.full[s], (g / FW_STAGES) & 1)) { atomicExch(&p.flags[0], 1); go = false; break; }
                    tc_fence_after();
                    const uint32_t a0 = smem_u32(A + kb * A_BLOCK), b0 = smem_u32(ring + s * W_BLOCK);
                    const int nj = l == 0 && kb == 1 ? (FW_K1 - 64) / 16 : 4;
                    for (int j = 0; j < nj; ++j)
                        mma_bf16(acc, sw128_desc(a0 + j * 32), sw128_desc(b0 + j * 32), idesc, (kb | j) != 0);
                    mma_commit(&p.empty[s]);
                }
                if (st) bulk_store_read();                 // the operand may be overwritten after this layer
                if (go) mma_commit(&p.tfull[b]);
            }
        }
        p.flags[2] = g;
        mma_commit(&p.done);
    } else if (warp >= 2) {
        const int q = warp & 3, half = (warp - 2) >> 2, et = threadIdx.x - 64;
        const int r = q * 32 + lane;                       // row of the tile
        const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
        float* sc = reinterpret_cast<float*>(scratch + (warp - 2) * FW_SCRATCH);
        const bool xvec = (reinterpret_cast<uintptr_t>(f.x) & 15u) == 0;
        const bool tvec = (reinterpret_cast<uintptr_t>(f.theta) & 7u) == 0;
        const bool ovec = ((reinterpret_cast<uintptr_t>(f.mean) | reinterpret_cast<uintptr_t>(f.sd)) & 7u) == 0;
        int layer = 0;
        bool go = true;
        for (int u = blockIdx.x; u < units && go; u += gridDim.x) {
            const int m0 = (u / f.groups) * TILE_M, t0 = (u % f.groups) * tpu;
            const int row = m0 + r;
            const bool store = TRAIN && t0 == 0;
            // the inputs as BF16 operand, rows beyond n and columns 72..79
            // zero (all loads in flight, then the stores)
            constexpr int XQ = FW_K1 / 4, XN = TILE_M * XQ / EPI_THREADS;
            static_assert(TILE_M * XQ % EPI_THREADS == 0, "whole rounds");
            float4 xv[XN];
#pragma unroll
            for (int e = 0; e < XN; ++e) {
                const int rr = (et + e * EPI_THREADS) / XQ, k = 4 * ((et + e * EPI_THREADS) % XQ);
                xv[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (m0 + rr < f.n && k < MLP_NIN) {
                    const float* src = f.x + (size_t)(m0 + rr) * MLP_NIN + k;
                    if (xvec) xv[e] = __ldg(reinterpret_cast<const float4*>(src));
                    else xv[e] = make_float4(src[0], src[1], src[2], src[3]);
                }
            }
#pragma unroll
            for (int e = 0; e < XN; ++e) {
                const int rr = (et + e * EPI_THREADS) / XQ, k = 4 * ((et + e * EPI_THREADS) % XQ);
                bf16 h[4] = { __float2bfloat16_rn(xv[e].x), __float2bfloat16_rn(xv[e].y),
                              __float2bfloat16_rn(xv[e].z), __float2bfloat16_rn(xv[e].w) };
                const uint2 w = *reinterpret_cast<const uint2*>(h);
                *reinterpret_cast<uint2*>(A + (k >> 6) * A_BLOCK + sw_off(rr, (k & 63) >> 3) + ((k & 4) ? 8 : 0)) = w;
                if (store && k < MLP_NIN)
                    *reinterpret_cast<uint2*>(f.X + (size_t)(m0 + rr) * MLP_D0 + k) = w;
            }
            fence_proxy_async_smem();
            mbar_arrive(&p.aready);
            // hidden layers: bias, ReLU, BF16 -> the next operand
            for (int l = 0; l < 2 && go; ++l, ++layer) {
                const int b = layer & 1;
                const bool ok = mbar_wait(&p.tfull[b], (layer >> 1) & 1);
                if (!epilogue_go(p, ok)) { atomicExch(&p.flags[0], 1); go = false; break; }
                tc_fence_after();
                uint32_t pos[4] = { 0u, 0u, 0u, 0u };      // positive activations of this lane's 128 columns
#pragma unroll
                for (int ch = 0; ch < 8; ++ch) {
                    const int c = half * 128 + 16 * ch;
                    float v[16], bi[16];
                    tmem_ld16(trow + (uint32_t)(b * 256 + c), v);
                    load16(bias + l * MLP_HID + c, bi);
                    __align__(16) bf16 h[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        h[i] = __float2bfloat16_rn(fmaxf(v[i] + bi[i], 0.0f));
                        if (TRAIN && (__bfloat16_as_ushort(h[i]) & 0x7FFFu)) pos[ch >> 1] |= 1u << (16 * (ch & 1) + i);
                    }
                    put_row16(A, r, c, h);
                }
                if (store) f.mask[((size_t)l * f.n + row) * 2 + half] = make_uint4(pos[0], pos[1], pos[2], pos[3]);
                tc_fence_before();
                mbar_arrive(&p.tempty[b]);
                fence_proxy_async_smem();
                mbar_arrive(&p.aready);
            }
            // output tiles: columns 0..127 means, 128..255 log-stds; this
            // warp's 64 parameters in two chunks of 32
            for (int t = t0; t < t0 + tpu && go; ++t, ++layer) {
                const int b = layer & 1, p0 = t * MLP_TP + half * 64;      // first parameter of this warp
                float2 th[16];
                if constexpr (TRAIN) fetch_rows(f.theta, tvec, m0 + q * 32, f.n, p0, lane, th);
                const bool ok = mbar_wait(&p.tfull[b], (layer >> 1) & 1);
                if (!epilogue_go(p, ok)) { atomicExch(&p.flags[0], 1); go = false; break; }
                tc_fence_after();
                float loss = 0.0f;
                const float scale = 1.0f / ((float)f.n * (float)MLP_NTH);
#pragma unroll
                for (int ch = 0; ch < 2; ++ch) {
                    const int i0 = p0 + 32 * ch;           // first parameter of the chunk
                    uint32_t gm[16], gl[16];               // TRAIN: BF16 gradients of this lane's row
                    float sd[TRAIN ? 1 : 32];
                    if constexpr (TRAIN) {
                        rows_to_scratch(sc, lane, th);
                        if (ch == 0) fetch_rows(f.theta, tvec, m0 + q * 32, f.n, p0 + 32, lane, th);
                        __syncwarp();
                    }
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        const int c = half * 64 + 32 * ch + 16 * s;
                        float mu[16], raw[16], bi[16];
                        tmem_ld16(trow + (uint32_t)(b * 256 + c), mu);
                        load16(bias + 2 * MLP_HID + i0 + 16 * s, bi);
#pragma unroll
                        for (int i = 0; i < 16; ++i) mu[i] += bi[i];
                        tmem_ld16(trow + (uint32_t)(b * 256 + MLP_TP + c), raw);
                        load16(bias + 2 * MLP_HID + MLP_D3 / 2 + i0 + 16 * s, bi);
#pragma unroll
                        for (int i = 0; i < 16; ++i) raw[i] += bi[i];
                        if constexpr (!TRAIN) {
#pragma unroll
                            for (int i = 0; i < 16; i += 2) {
                                *reinterpret_cast<float2*>(sc + lane * SC_F32 + 16 * s + i) = make_float2(mu[i], mu[i + 1]);
                                sd[16 * s + i] = expf(fminf(fmaxf(raw[i], f.ls_min), f.ls_max));
                                sd[16 * s + i + 1] = expf(fminf(fmaxf(raw[i + 1], f.ls_min), f.ls_max));
                            }
                        } else {
                            // Gaussian negative log-likelihood and its
                            // gradient (mean over n x 450), BF16
                            bf16 hm[2], hl[2];
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const float2 tv = *reinterpret_cast<const float2*>(sc + lane * SC_F32 + 16 * s + (i & ~1));
                                const float ls = fminf(fmaxf(raw[i], f.ls_min), f.ls_max);
                                const float rr = ((i & 1) ? tv.y : tv.x) - mu[i];
                                const float e2 = expf(-2.0f * ls);
                                if (i0 + 16 * s + i < MLP_NTH) loss += ls + 0.5f * rr * rr * e2;
                                const float dmu = -rr * e2 * scale;
                                const float dls = (raw[i] > f.ls_min && raw[i] < f.ls_max) ? (1.0f - rr * rr * e2) * scale
                                                                                           : 0.0f;
                                hm[i & 1] = __float2bfloat16_rn(dmu);
                                hl[i & 1] = __float2bfloat16_rn(dls);
                                if (i & 1) {
                                    gm[8 * s + i / 2] = *reinterpret_cast<const uint32_t*>(hm);
                                    gl[8 * s + i / 2] = *reinterpret_cast<const uint32_t*>(hl);
                                }
                            }
                        }
                    }
                    __syncwarp();
                    if constexpr (!TRAIN) {
                        scratch_to_rows(sc, f.mean, ovec, m0 + q * 32, f.n, i0, lane);
                        __syncwarp();
#pragma unroll
                        for (int i = 0; i < 32; i += 2)
                            *reinterpret_cast<float2*>(sc + lane * SC_F32 + i) = make_float2(sd[i], sd[i + 1]);
                        __syncwarp();
                        scratch_to_rows(sc, f.sd, ovec, m0 + q * 32, f.n, i0, lane);
                        __syncwarp();
                    } else {
                        // dY columns i0 .. and 450 + i0 .. (the padding columns
                        // 900.. stay zero): sixteen 32-bit words a row, two
                        // rows at a time
                        uint32_t* sw = reinterpret_cast<uint32_t*>(sc);
#pragma unroll
                        for (int i = 0; i < 16; i += 2) {
                            *reinterpret_cast<uint2*>(sw + lane * SC_BF16 + i) = make_uint2(gm[i], gm[i + 1]);
                            *reinterpret_cast<uint2*>(sw + (32 + lane) * SC_BF16 + i) = make_uint2(gl[i], gl[i + 1]);
                        }
                        __syncwarp();
                        if (i0 + 2 * (lane & 15) < MLP_NTH) {
                            uint32_t* o = reinterpret_cast<uint32_t*>(f.dY + (size_t)(m0 + q * 32) * MLP_D3 + i0) +
                                          (lane & 15);
#pragma unroll
                            for (int k = 0; k < 16; ++k) {
                                const int rr = 2 * k + (lane >> 4);
                                o[(size_t)rr * (MLP_D3 / 2)] = sw[rr * SC_BF16 + (lane & 15)];
                                o[(size_t)rr * (MLP_D3 / 2) + MLP_NTH / 2] = sw[(32 + rr) * SC_BF16 + (lane & 15)];
                            }
                        }
                        __syncwarp();
                    }
                }
                tc_fence_before();
                mbar_arrive(&p.tempty[b]);
                if constexpr (TRAIN) {
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
                    if (lane == 0) f.loss_part[((m0 / TILE_M) * 4 + t) * 8 + (warp - 2)] = loss * scale;
                }
            }
        }
    }
    pipe_end(p, tmem, f.err);
}

// ------------------------------------------------------------------ backward
constexpr int BW_STAGES = 3;
constexpr int BW_STAGE = A_BLOCK + W_BLOCK;
constexpr int BW_SMEM = 4 * A_BLOCK + BW_STAGES * BW_STAGE + 1024 + (int)sizeof(Pipe<BW_STAGES>);

// Per row tile: dZ2 = (dY W3) where H2 > 0 (K = 1024; dY K-major, W3 as it is
// stored, MN-major), which becomes the operand of dZ1 = (dZ2 W2) where H1 > 0.
// Both go to global memory from the operand buffer.
__global__ void __launch_bounds__(THREADS, 1)
mlp_backward_kernel(const __grid_constant__ MlpBackwardMaps maps, const MlpBackward f)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* A = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* ring = A + 4 * A_BLOCK;
    Pipe<BW_STAGES>& p = *reinterpret_cast<Pipe<BW_STAGES>*>(ring + BW_STAGES * BW_STAGE);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem = pipe_init(p);
    wait_for_previous();                       // the forward pass
    start_next();
    const int tiles = f.n / TILE_M;
    constexpr int NK = MLP_D3 / 64 + MLP_HID / 64;         // K blocks of the two products

    if (warp == 0 && lane == 0) {
        int g = 0;
        bool go = true;
        for (int u = blockIdx.x; u < tiles && go; u += gridDim.x) {
            for (int k = 0; k < NK; ++k) {
                if (!(go = stage_free(p, g))) break;
                const int s = g % BW_STAGES;
                uint8_t* st = ring + s * BW_STAGE;
                const bool first = k < MLP_D3 / 64;
                mbar_expect_tx(&p.full[s], first ? BW_STAGE : W_BLOCK);
                if (first) tma_load_2d(st, &maps.dy, k * 64, u * TILE_M, &p.full[s]);
                // 64 rows of K by 256 columns, in 64-column boxes
                for (int c = 0; c < 4; ++c)
                    tma_load_2d(st + A_BLOCK + c * 8192, first ? &maps.w3 : &maps.w2, c * 64,
                                (first ? k : k - MLP_D3 / 64) * 64, &p.full[s]);
                ++g;
            }
        }
        p.flags[1] = g;
    } else if (warp == 1 && lane == 0) {
        // MMA issuer; it also stores dZ2 and dZ1 from the operand buffer
        constexpr uint32_t idesc = mma_idesc(256, false, true);
        int g = 0, layer = 0, ready = 0;
        bool go = true;
        for (int u = blockIdx.x; u < tiles && go; u += gridDim.x) {
            // l = 0, 1: the products (the second's operand is dZ2); l = 2: dZ1
            // is ready
            for (int l = 0; l < 3 && go; ++l) {
                const int b = layer & 1;
                bool ok = l == 2 || mbar_wait(&p.tempty[b], ((layer >> 1) & 1) ^ 1);
                if (l > 0) ok = ok && mbar_wait(&p.aready, ready++ & 1);
                if (!ok || aborted(p)) { atomicExch(&p.flags[0], 1); go = false; break; }
                tc_fence_after();
                if (l > 0) {
                    for (int kb = 0; kb < 4; ++kb)
                        tma_store_2d(l == 1 ? &maps.dz2 : &maps.dz1, A + kb * A_BLOCK, kb * 64, u * TILE_M);
                    bulk_store_commit();
                }
                if (l < 2) {
                    const uint32_t acc = tmem + (uint32_t)(b * 256);
                    const int nk = l == 0 ? MLP_D3 / 64 : MLP_HID / 64;
                    for (int kb = 0; kb < nk; ++kb, ++g) {
                        const int s = g % BW_STAGES;
                        if (!mbar_wait(&p.full[s], (g / BW_STAGES) & 1)) { atomicExch(&p.flags[0], 1); go = false; break; }
                        tc_fence_after();
                        const uint32_t b0 = smem_u32(ring + s * BW_STAGE + A_BLOCK);
                        const uint32_t a0 = l == 0 ? smem_u32(ring + s * BW_STAGE) : smem_u32(A + kb * A_BLOCK);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            mma_bf16(acc, sw128_desc(a0 + j * 32), sw128_mn_desc(b0 + j * 2048, 8192), idesc,
                                     (kb | j) != 0);
                        mma_commit(&p.empty[s]);
                    }
                }
                if (l > 0) bulk_store_read();              // the operand buffer may be overwritten after this
                if (l < 2) {
                    if (go) mma_commit(&p.tfull[b]);
                    ++layer;
                }
            }
        }
        p.flags[2] = g;
        mma_commit(&p.done);
    } else if (warp >= 2) {
        const int q = warp & 3, half = (warp - 2) >> 2;
        const int r = q * 32 + lane;
        const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
        int layer = 0;
        bool go = true;
        for (int u = blockIdx.x; u < tiles && go; u += gridDim.x) {
            const int row = u * TILE_M + r;
            for (int l = 0; l < 2 && go; ++l, ++layer) {
                const int b = layer & 1;
                // the activations' signs mask the gradient: layer 2's, then layer 1's
                const uint4 mk = __ldg(f.mask + ((size_t)(1 - l) * f.n + row) * 2 + half);
                const uint32_t pos[4] = { mk.x, mk.y, mk.z, mk.w };
                const bool ok = mbar_wait(&p.tfull[b], (layer >> 1) & 1);
                if (!epilogue_go(p, ok)) { atomicExch(&p.flags[0], 1); go = false; break; }
                tc_fence_after();
#pragma unroll
                for (int ch = 0; ch < 8; ++ch) {
                    const int c = half * 128 + 16 * ch;
                    float v[16];
                    __align__(16) bf16 h[16];
                    tmem_ld16(trow + (uint32_t)(b * 256 + c), v);
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        h[i] = __float2bfloat16_rn(((pos[ch >> 1] >> (16 * (ch & 1) + i)) & 1u) ? v[i] : 0.0f);
                    put_row16(A, r, c, h);
                }
                tc_fence_before();
                mbar_arrive(&p.tempty[b]);
                fence_proxy_async_smem();
                mbar_arrive(&p.aready);
            }
        }
    }
    pipe_end(p, tmem, f.err);
}

// ------------------------------------------------------------------ weight gradients
constexpr int GR_STAGES = 4;
constexpr int GR_STAGE = A_BLOCK + W_BLOCK;
constexpr int GR_SMEM = GR_STAGES * GR_STAGE + 1024 + (int)sizeof(Pipe<GR_STAGES>);
// row tiles of product k (dW3, dW2, dW1), each 128 x (256, 256, 128)
__host__ __device__ constexpr int gr_tiles(int k) { return (k == 0 ? MLP_D3 : MLP_HID) / 128; }

// One launch for the three products dW = dZ^T H over the batch, both
// operands row-major as stored (MN-major).  A unit is a row tile of one
// product and a slice of the batch's K blocks; dW3's units, the longest,
// come first.
__global__ void __launch_bounds__(THREADS, 1)
mlp_grad_kernel(const __grid_constant__ MlpGradMaps maps, const MlpGrads f)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Pipe<GR_STAGES>& p = *reinterpret_cast<Pipe<GR_STAGES>*>(ring + GR_STAGES * GR_STAGE);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem = pipe_init(p);
    const int u1 = gr_tiles(0) * f.splits[0], u2 = u1 + gr_tiles(1) * f.splits[1];
    const int units = u2 + gr_tiles(2) * f.splits[2], nkb = f.n / 64;
    struct Unit {
        int k, m0, bn, z, k0, k1;
    };
    const auto unit = [&](int u) {
        Unit x;
        x.k = u < u1 ? 0 : u < u2 ? 1 : 2;
        u -= x.k == 0 ? 0 : x.k == 1 ? u1 : u2;
        const int tiles = gr_tiles(x.k);
        x.m0 = u % tiles * 128;
        x.z = u / tiles;
        x.bn = x.k == 2 ? 128 : 256;
        const int nk = nkb / (x.k == 0 ? f.splits[0] : x.k == 1 ? f.splits[1] : f.splits[2]);
        x.k0 = x.z * nk;
        x.k1 = x.k0 + nk;
        return x;
    };

    if (warp == 0 && lane == 0) {
        // dW3's operands are the forward pass's, complete before the backward
        // pass let this kernel start; the others wait for the backward pass
        int g = 0;
        bool go = true, waited = false;
        for (int u = blockIdx.x; u < units && go; u += gridDim.x) {
            const Unit x = unit(u);
            if (x.k != 0 && !waited) {
                wait_for_previous();
                start_next();
                waited = true;
            }
            for (int kb = x.k0; kb < x.k1; ++kb) {
                if (!(go = stage_free(p, g))) break;
                const int s = g % GR_STAGES;
                uint8_t* st = ring + s * GR_STAGE;
                mbar_expect_tx(&p.full[s], A_BLOCK + x.bn * 128);
                for (int c = 0; c < 2; ++c) tma_load_2d(st + c * 8192, &maps.a[x.k], x.m0 + c * 64, kb * 64, &p.full[s]);
                for (int c = 0; c < x.bn / 64; ++c)
                    tma_load_2d(st + A_BLOCK + c * 8192, &maps.b[x.k], c * 64, kb * 64, &p.full[s]);
                ++g;
            }
        }
        if (!waited) {
            wait_for_previous();
            start_next();
        }
        p.flags[1] = g;
    } else if (warp == 1 && lane == 0) {
        int g = 0, i = 0;
        bool go = true;
        for (int u = blockIdx.x; u < units && go; u += gridDim.x, ++i) {
            const Unit x = unit(u);
            const int b = i & 1;
            const uint32_t idesc = x.bn == 256 ? mma_idesc(256, true, true) : mma_idesc(128, true, true);
            if (!mbar_wait(&p.tempty[b], ((i >> 1) & 1) ^ 1) || aborted(p)) { atomicExch(&p.flags[0], 1); break; }
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)(b * 256);
            for (int kb = x.k0; kb < x.k1; ++kb, ++g) {
                const int s = g % GR_STAGES;
                if (!mbar_wait(&p.full[s], (g / GR_STAGES) & 1)) { atomicExch(&p.flags[0], 1); go = false; break; }
                tc_fence_after();
                const uint32_t a0 = smem_u32(ring + s * GR_STAGE), b0 = a0 + A_BLOCK;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    mma_bf16(acc, sw128_mn_desc(a0 + j * 2048, 8192), sw128_mn_desc(b0 + j * 2048, 8192), idesc,
                             kb > x.k0 || j > 0);
                mma_commit(&p.empty[s]);
            }
            if (go) mma_commit(&p.tfull[b]);
        }
        p.flags[2] = g;
        mma_commit(&p.done);
    } else if (warp >= 2) {
        const int q = warp & 3, half = (warp - 2) >> 2;
        const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
        int i = 0;
        for (int u = blockIdx.x; u < units; u += gridDim.x, ++i) {
            const Unit x = unit(u);
            const int b = i & 1;
            const bool ok = mbar_wait(&p.tfull[b], (i >> 1) & 1);
            if (!epilogue_go(p, ok)) { atomicExch(&p.flags[0], 1); break; }
            tc_fence_after();
            const int rows = x.k == 0 ? MLP_D3 : MLP_HID;
            float* out = f.part[x.k] + ((size_t)x.z * rows + x.m0 + q * 32 + lane) * x.bn;
#pragma unroll 1
            for (int c = half * (x.bn / 2); c < (half + 1) * (x.bn / 2); c += 16) {
                float v[16];
                tmem_ld16(trow + (uint32_t)(b * 256 + c), v);
                store_32b(out + c, v);
                store_32b(out + c + 8, v + 8);
            }
            tc_fence_before();
            mbar_arrive(&p.tempty[b]);
        }
    }
    pipe_end(p, tmem, f.err);
}

template <typename Fn>
cudaError_t smem_opt(Fn fn, int bytes)
{
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

}  // namespace

int mlp_sm_count()
{
    int dev = 0, c = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || c <= 0) c = 148;
    return c;
}

// Slices of each weight gradient: doubled while the CTAs of the product
// alone stay within about one wave of the 152 SMs and every slice keeps two K
// blocks or more (the sums over slices are part of the results, so the
// slicing is fixed by the batch alone).
void mlp_grad_splits(int n, int splits[3])
{
    const int nk = n / 64;
    for (int k = 0; k < 3; ++k) {
        int sp = 1;
        while (2 * sp * gr_tiles(k) <= 160 && nk % (2 * sp) == 0 && nk / (2 * sp) >= 2) sp *= 2;
        splits[k] = sp;
    }
}

int mlp_groups(int n, int sms)
{
    const int tiles = (n + TILE_M - 1) / TILE_M;
    return 4 * tiles <= sms ? 4 : 2 * tiles <= sms ? 2 : 1;
}

cudaError_t launch_mlp_forward(const MlpForwardMaps& m, const MlpForward& f, cudaStream_t s)
{
    const int units = (f.n + TILE_M - 1) / TILE_M * f.groups, grid = std::min(units, mlp_sm_count());
    cudaError_t e = f.theta ? smem_opt(mlp_forward_kernel<true>, FW_SMEM) : smem_opt(mlp_forward_kernel<false>, FW_SMEM);
    if (e != cudaSuccess) return e;
    if (f.theta) mlp_forward_kernel<true><<<grid, THREADS, FW_SMEM, s>>>(m, f);
    else mlp_forward_kernel<false><<<grid, THREADS, FW_SMEM, s>>>(m, f);
    return cudaGetLastError();
}

cudaError_t launch_mlp_backward(const MlpBackwardMaps& m, const MlpBackward& b, cudaStream_t s)
{
    cudaError_t e = smem_opt(mlp_backward_kernel, BW_SMEM);
    if (e != cudaSuccess) return e;
    return launch_dependent(mlp_backward_kernel, std::min(b.n / TILE_M, mlp_sm_count()), THREADS, BW_SMEM, s, m, b);
}

cudaError_t launch_mlp_grads(const MlpGradMaps& m, const MlpGrads& g, cudaStream_t s)
{
    cudaError_t e = smem_opt(mlp_grad_kernel, GR_SMEM);
    if (e != cudaSuccess) return e;
    const int units = gr_tiles(0) * g.splits[0] + gr_tiles(1) * g.splits[1] + gr_tiles(2) * g.splits[2];
    return launch_dependent(mlp_grad_kernel, std::min(units, mlp_sm_count()), THREADS, GR_SMEM, s, m, g);
}

}  // namespace npp
