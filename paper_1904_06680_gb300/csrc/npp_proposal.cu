// npp_proposal.cu -- the learned sampling proposal: scene encoding, the
// 72-256-256-900 network on BF16 tensor-core GEMMs (forward, backward),
// Gaussian negative log-likelihood, Adam, and the standalone GEMM entry.
//
// The paper samples theta ~ N(0, I) every sampling time (Sect. II-D
// "Fourth") and lists guiding the sampling as future work (Sect. V); this
// file is that guide, built so that it never bends the method: its output
// (mean, std) only feeds npp_plan_step_proposal, whose proposal samples
// are mixed with isotropic ones and judged by the exact rollout cost.
//
// Layout of the FP32 master parameters (padded for the tensor-core tiles):
//   W1 [256][128] (inputs 72..127 zero), b1 [256], W2 [256][256], b2 [256],
//   W3 [1024][256] (rows 900..1023 zero), b3 [1024]
// BF16 copies W1, W2, W3 and W3 in the forward pass's row order (W3f) are
// refreshed by every update.
//
// A training step is four launches: the forward pass with the loss and its
// gradient, the activations' gradients, the weight gradients (npp_mlp.cu) and
// the update below.
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/npp_proposal.h"
#include "npp_gemm.cuh"
#include "npp_internal.h"
#include "npp_launch.cuh"
#include "npp_mlp.cuh"

using namespace npp;

namespace {

constexpr int NIN_X = MLP_NIN;
constexpr int D0 = MLP_D0;
constexpr int HID = MLP_HID;
constexpr int NTH = MLP_NTH;
constexpr int D3 = MLP_D3;
constexpr int NBINS = 64;
constexpr float R_HIST = 20.0f;

// offsets into the flat master / gradient / moment buffers
constexpr size_t OFF_W1 = 0;
constexpr size_t OFF_B1 = OFF_W1 + (size_t)HID * D0;
constexpr size_t OFF_W2 = OFF_B1 + HID;
constexpr size_t OFF_B2 = OFF_W2 + (size_t)HID * HID;
constexpr size_t OFF_W3 = OFF_B2 + HID;
constexpr size_t OFF_B3 = OFF_W3 + (size_t)D3 * HID;
constexpr size_t N_FLAT = OFF_B3 + D3;
// packed (unpadded) parameter count of the public layout
constexpr int N_PACKED = HID * NIN_X + HID + HID * HID + HID + 2 * NTH * HID + 2 * NTH;

using bf16 = __nv_bfloat16;

// ------------------------------------------------------------------ encoding
// One block per scene: nearness-weighted polar histogram of the points in
// the EV-aligned frame at t (fixed-point sums, so the result does not
// depend on the order of the atomic adds), squashed h / (1 + h), then the
// rollout's 8 network inputs at h = 0.
// A weight is a multiple of 2^-32; its upper and lower 16 bits are summed
// apart (32-bit shared atomics, which the hardware does in place; 64-bit ones
// loop), without overflow up to 65535 points; beyond, the upper sums carry
// into a third word.
// Bound: latency (reads, atan2, atomics); ENC_AHEAD points a thread in flight.
// Encoding and forward pass of 300 scenes on GB300: 33 -> 28.5 us (256
// threads, one point at a time and 64-bit atomics before).
constexpr int ENC_THREADS = 512;
constexpr int ENC_AHEAD = 4;
__global__ void __launch_bounds__(ENC_THREADS) encode_kernel(const DevCfg c, const npp_scene* __restrict__ scenes,
                                                             const float4* __restrict__ obs, float* __restrict__ x)
{
    __shared__ unsigned lo[NBINS], hi[NBINS], over[NBINS];
    const npp_scene& sc = scenes[blockIdx.x];
    for (int k = threadIdx.x; k < NBINS; k += ENC_THREADS) lo[k] = hi[k] = over[k] = 0u;
    __syncthreads();
    float s0, c0;
    sincosf(sc.state.phi, &s0, &c0);
    const float4* p = obs + sc.obs_offset;
    const int M = sc.M;
    const bool large = M > 65535;
    for (int j0 = threadIdx.x; j0 < M; j0 += ENC_AHEAD * ENC_THREADS) {
        float4 o[ENC_AHEAD];
#pragma unroll
        for (int u = 0; u < ENC_AHEAD; ++u) {
            const int j = j0 + u * ENC_THREADS;
            o[u] = p[j < M ? j : j0];
        }
#pragma unroll
        for (int u = 0; u < ENC_AHEAD; ++u) {
            float px, py, vx, vy;
            ev_point(o[u], sc.state.x, sc.state.y, s0, c0, px, py, vx, vy);
            const float d = sqrtf(fmaf(px, px, py * py));
            const float w = 1.0f - d / R_HIST;
            if (j0 + u * ENC_THREADS < M && w > 0.0f) {
                const float t = (atan2f(py, px) + 3.14159265358979323846f) * (NBINS / 6.28318530717958647692f);
                const int k = min(max((int)floorf(t), 0), NBINS - 1);
                const unsigned long long v = __float2ull_rn(w * 4294967296.0f);
                const unsigned l = (unsigned)(v & 0xFFFFu), h = (unsigned)(v >> 16);
                const unsigned was_l = atomicAdd(&lo[k], l);
                const unsigned was_h = atomicAdd(&hi[k], h);
                if (large) {
                    // carries of the two sums (2^32 of lo is 2^16 of hi)
                    if (was_l + l < was_l && atomicAdd(&hi[k], 65536u) > 0xFFFEFFFFu) atomicAdd(&over[k], 1u);
                    if (was_h + h < was_h) atomicAdd(&over[k], 1u);
                }
            }
        }
    }
    __syncthreads();
    float* xr = x + (size_t)blockIdx.x * NIN_X;
    for (int k = threadIdx.x; k < NBINS; k += ENC_THREADS) {
        const unsigned long long sum = ((unsigned long long)over[k] << 48) + ((unsigned long long)hi[k] << 16) + lo[k];
        const float h = (float)((double)sum * (1.0 / 4294967296.0));
        xr[k] = h / (1.0f + h);
    }
    if (threadIdx.x == 0) {
        const float gdx = sc.goal.x - sc.state.x, gdy = sc.goal.y - sc.state.y;
        const float gxi = c0 * gdx + s0 * gdy, geta = -s0 * gdx + c0 * gdy;
        float* s = xr + NBINS;
        s[0] = gxi * c.idxi;
        s[1] = geta * c.ideta;
        const float dph = sc.goal.phi - sc.state.phi;
        s[2] = (dph - 6.28318530717958647692f * floorf((dph + 3.14159265358979323846f) *
                                                       0.15915494309189533577f)) * c.idphi;
        s[3] = (sc.goal.v - sc.state.v) * c.idv;
        s[4] = sc.state.a_prev0;
        s[5] = sc.state.a_prev1;
        s[6] = sc.state.v * c.idv;
        s[7] = (float)sc.T * (1.0f / (float)sc.T);
    }
}

// BF16 copies of the weight matrices
__global__ void convert_kernel(const float* __restrict__ w, bf16* __restrict__ W1, bf16* __restrict__ W2,
                               bf16* __restrict__ W3, bf16* __restrict__ W3f)
{
    const int n1 = HID * D0, n2 = HID * HID, n3 = D3 * HID;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n1 + n2 + n3; t += gridDim.x * blockDim.x) {
        if (t < n1) W1[t] = __float2bfloat16_rn(w[OFF_W1 + t]);
        else if (t < n1 + n2) W2[t - n1] = __float2bfloat16_rn(w[OFF_W2 + t - n1]);
        else {
            const int u = t - n1 - n2, r = u / HID;
            const bf16 q = __float2bfloat16_rn(w[OFF_W3 + u]);
            W3[u] = q;
            if (r < 2 * NTH) W3f[(size_t)mlp_row(r) * HID + u % HID] = q;
        }
    }
}

// Adam with bias correction (c1, c2) on one parameter
struct Adam {
    float lr, b1, b2, eps, c1, c2;
};
__device__ __forceinline__ float adam_step(const Adam& a, float g, float w, float& m, float& v)
{
    // (every rounding written out: the updates are the same bits however the
    // step is compiled)
    m = fmaf(1.0f - a.b1, g, __fmul_rn(a.b1, m));
    v = fmaf(__fmul_rn(1.0f - a.b2, g), g, __fmul_rn(a.b2, v));
    const float mhat = __fdiv_rn(m, a.c1), vhat = __fdiv_rn(v, a.c2);
    return __fsub_rn(w, __fdiv_rn(__fmul_rn(a.lr, mhat), __fadd_rn(__fsqrt_rn(vhat), a.eps)));
}

// The end of a training step: gradients summed in a fixed order (weights
// over the batch slices; biases over the batch, lane l of 32 taking rows
// 8 l .. 8 l + 7 of every 256, then the lanes in a pairwise tree), Adam on
// the FP32 masters, BF16 copies, the loss.
// Blocks 0 .. UPD_B - 1: UPD_COLS biases each, the longest; then four weights
// a thread; the last block the loss.
// Bound: L2 reads of the partials (40 MB at batch 8192) and of the batch's
// gradients for the bias sums.  The weight gradients' kernel lets this one
// start once the backward pass is complete, so the biases and the loss, which
// need no more than that, are done while it runs; the weights wait for it.
// One launch instead of four (split sum, bias
// gradients, Adam, BF16 copies: 36 us of a 187 us step at batch 8192).
struct UpdateArgs {
    float *w, *m, *v, *g;
    bf16 *W[3], *W3f;                        // W1, W2, W3; W3 in the forward order
    const float* part[3];                    // dW1, dW2, dW3 partials
    int splits[3];
    const bf16* dz[3];                       // dZ1, dZ2, dY
    int batch;
    const float* loss_part;
    int n_loss;
    float* loss;
    Adam adam;
};
constexpr int UPD_THREADS = 256;
constexpr int UPD_COLS = 32;
constexpr int UPD_B = (D3 + 2 * HID) / UPD_COLS;
constexpr int UPD_W = (HID * D0 + HID * HID + D3 * HID) / 4 / UPD_THREADS;

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

__global__ void __launch_bounds__(UPD_THREADS) update_kernel(const UpdateArgs a)
{
    __shared__ float red[32][UPD_COLS + 1];
    const int tid = threadIdx.x;
    if (blockIdx.x < UPD_B) {
        // thread (lane l of the sum, four columns); 32 rows' loads in flight
        const int c0 = blockIdx.x * UPD_COLS, lc = tid % 8 * 4, l = tid / 8;
        const int k = c0 < HID ? 0 : c0 < 2 * HID ? 1 : 2;
        const int col = c0 - k * HID, width = k == 2 ? D3 : HID;
        const bf16* p = a.dz[k] + (size_t)(8 * l) * width + col + lc;
        float s[4] = { 0.f, 0.f, 0.f, 0.f };
        int r = 8 * l;
        for (; r + 3 * 256 < a.batch; r += 4 * 256, p += (size_t)4 * 256 * width) {
            uint2 t[32];
#pragma unroll
            for (int u = 0; u < 32; ++u)
                t[u] = __ldg(reinterpret_cast<const uint2*>(p + (size_t)((u >> 3) * 256 + (u & 7)) * width));
#pragma unroll
            for (int u = 0; u < 32; ++u) {
                s[0] += bf_lo(t[u].x); s[1] += bf_hi(t[u].x);
                s[2] += bf_lo(t[u].y); s[3] += bf_hi(t[u].y);
            }
        }
        for (; r < a.batch; r += 256, p += (size_t)256 * width) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const uint2 t = __ldg(reinterpret_cast<const uint2*>(p + (size_t)u * width));
                s[0] += bf_lo(t.x); s[1] += bf_hi(t.x);
                s[2] += bf_lo(t.y); s[3] += bf_hi(t.y);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) red[l][lc + j] = s[j];
        for (int off = 16; off > 0; off >>= 1) {
            __syncthreads();
            for (int e = tid; e < off * UPD_COLS; e += UPD_THREADS)
                red[e / UPD_COLS][e % UPD_COLS] += red[e / UPD_COLS + off][e % UPD_COLS];
        }
        __syncthreads();
        if (tid < UPD_COLS) {
            const float g = red[0][tid];
            const size_t i = (k == 0 ? OFF_B1 : k == 1 ? OFF_B2 : OFF_B3) + col + tid;
            float m = a.m[i], v = a.v[i];
            a.w[i] = adam_step(a.adam, g, a.w[i], m, v);
            a.g[i] = g; a.m[i] = m; a.v[i] = v;
        }
    } else if (blockIdx.x < UPD_B + UPD_W) {
        constexpr int n1 = HID * D0 / 4, n2 = HID * HID / 4, n3 = D3 * HID / 4;
        int i = (blockIdx.x - UPD_B) * UPD_THREADS + tid;
        const int k = i < n1 ? 0 : i < n1 + n2 ? 1 : 2;
        i -= k == 0 ? 0 : k == 1 ? n1 : n1 + n2;
        wait_for_previous();                     // the weight gradients
        const size_t size = k == 0 ? n1 : k == 1 ? n2 : n3;
        const size_t off = k == 0 ? OFF_W1 : k == 1 ? OFF_W2 : OFF_W3;
        const float4* p = reinterpret_cast<const float4*>(a.part[k]) + i;
        const int S = a.splits[k];
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        int z = 0;
        for (; z + 16 <= S; z += 16) {           // sixteen loads in flight, added in slice order
            float4 t[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) t[u] = p[(size_t)(z + u) * size];
#pragma unroll
            for (int u = 0; u < 16; ++u) { g.x += t[u].x; g.y += t[u].y; g.z += t[u].z; g.w += t[u].w; }
        }
        for (; z < S; ++z) {
            const float4 t = p[(size_t)z * size];
            g.x += t.x; g.y += t.y; g.z += t.z; g.w += t.w;
        }
        float4* G = reinterpret_cast<float4*>(a.g + off) + i;
        float4* W = reinterpret_cast<float4*>(a.w + off) + i;
        float4* M = reinterpret_cast<float4*>(a.m + off) + i;
        float4* V = reinterpret_cast<float4*>(a.v + off) + i;
        float4 w = *W, m = *M, v = *V;
        w.x = adam_step(a.adam, g.x, w.x, m.x, v.x);
        w.y = adam_step(a.adam, g.y, w.y, m.y, v.y);
        w.z = adam_step(a.adam, g.z, w.z, m.z, v.z);
        w.w = adam_step(a.adam, g.w, w.w, m.w, v.w);
        *G = g; *W = w; *M = m; *V = v;
        bf16 h[4] = { __float2bfloat16_rn(w.x), __float2bfloat16_rn(w.y), __float2bfloat16_rn(w.z),
                      __float2bfloat16_rn(w.w) };
        const uint2 q = *reinterpret_cast<const uint2*>(h);
        reinterpret_cast<uint2*>(a.W[k])[i] = q;
        const int r = i / (HID / 4);
        if (k == 2 && r < 2 * NTH) reinterpret_cast<uint2*>(a.W3f)[mlp_row(r) * (HID / 4) + i % (HID / 4)] = q;
    } else {
        float s = 0.0f;
        for (int i = tid; i < a.n_loss; i += UPD_THREADS) s += a.loss_part[i];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if ((tid & 31) == 0) red[tid >> 5][0] = s;
        __syncthreads();
        if (tid == 0) {
            float t = 0.0f;
            for (int j = 0; j < UPD_THREADS / 32; ++j) t += red[j][0];
            *a.loss = t;
        }
    }
}

__device__ int g_gemm_err;

std::string g_prop_err;

npp_status perr(npp_status s, const std::string& msg)
{
    g_prop_err = msg;
    set_global_error(msg.c_str());
    return s;
}

}  // namespace

struct npp_proposal {
    npp_proposal_config cfg;
    int B;
    int t;                                  // Adam steps taken
    float* w; float* m; float* v; float* g; // flat FP32 [N_FLAT]
    bf16 *W1, *W2, *W3, *W3f;               // W3f: W3 in the forward pass's row order
    bf16 *X, *H1, *H2, *dY, *dZ2, *dZ1;     // activations and their gradients, row-major [batch][..]
    float* packed;                          // staging of parameter and gradient reads, [N_PACKED]
    std::mutex packed_lock;
    float* loss;                            // scratch loss when the caller passes none
    int* err;
    int splits[3];                          // batch slices of the weight gradients
    float* part[3];                         // their partials: dW3, dW2, dW1
    float* loss_part;
    uint4* mask;                            // bits of the positive activations
    MlpForwardMaps fmaps;
    MlpBackwardMaps bmaps;
    MlpGradMaps grads;
};

namespace {

MlpForward forward_args(const npp_proposal* P, const float* x, int n)
{
    MlpForward f;
    memset(&f, 0, sizeof f);
    f.x = x;
    f.n = n;
    f.b1 = P->w + OFF_B1; f.b2 = P->w + OFF_B2; f.b3 = P->w + OFF_B3;
    f.ls_min = P->cfg.ls_min; f.ls_max = P->cfg.ls_max;
    f.groups = mlp_groups(n, mlp_sm_count());
    f.err = P->err;
    return f;
}

cudaError_t refresh_bf16(npp_proposal* P, cudaStream_t s)
{
    convert_kernel<<<512, 256, 0, s>>>(P->w, P->W1, P->W2, P->W3, P->W3f);
    return cudaGetLastError();
}

// packed public layout <-> padded flat layout
void packed_to_flat(const float* src, float* flat)
{
    std::memset(flat, 0, N_FLAT * sizeof(float));
    size_t o = 0;
    for (int r = 0; r < HID; ++r)
        for (int k = 0; k < NIN_X; ++k) flat[OFF_W1 + (size_t)r * D0 + k] = src[o++];
    for (int r = 0; r < HID; ++r) flat[OFF_B1 + r] = src[o++];
    for (int i = 0; i < HID * HID; ++i) flat[OFF_W2 + i] = src[o++];
    for (int r = 0; r < HID; ++r) flat[OFF_B2 + r] = src[o++];
    for (int i = 0; i < 2 * NTH * HID; ++i) flat[OFF_W3 + i] = src[o++];
    for (int r = 0; r < 2 * NTH; ++r) flat[OFF_B3 + r] = src[o++];
}

// padded flat layout -> packed public layout, on the device (one copy of what
// the caller gets instead of a copy of the padded layout and a host loop over
// it: 16 training steps and two reads took 1787 us, now 1637)
__global__ void pack_flat_kernel(const float* __restrict__ flat, float* __restrict__ packed)
{
    constexpr int p1 = HID * NIN_X;
    constexpr int w3 = HID + HID * HID + HID, b3 = w3 + 2 * NTH * HID;      // offsets into the rest
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N_PACKED; i += gridDim.x * blockDim.x) {
        const int j = i - p1;
        size_t o;
        if (j < 0) o = OFF_W1 + (size_t)(i / NIN_X) * D0 + i % NIN_X;
        else if (j < b3) o = OFF_B1 + j;                 // b1, W2, b2, W3's rows follow one another
        else o = OFF_B3 + (j - b3);
        packed[i] = flat[o];
    }
}

npp_status read_flat(npp_proposal* P, const float* dev, float* host_packed)
{
    std::lock_guard<std::mutex> lock(P->packed_lock);      // threads that read share the staging
    pack_flat_kernel<<<(N_PACKED + 511) / 512, 512>>>(dev, P->packed);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpy(host_packed, P->packed, (size_t)N_PACKED * 4, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return perr(NPP_CUDA_ERROR, std::string("proposal read: ") + cudaGetErrorString(e));
    int err = 0;
    e = cudaMemcpy(&err, P->err, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return perr(NPP_CUDA_ERROR, std::string("proposal read: ") + cudaGetErrorString(e));
    if (err) return perr(NPP_DEVICE_TIMEOUT, "a proposal GEMM pipeline wait timed out");
    return NPP_OK;
}

}  // namespace

extern "C" {

int32_t npp_proposal_n_params(void) { return N_PACKED; }

npp_status npp_proposal_create(const npp_proposal_config* cfg, npp_proposal** out)
{
    if (!cfg || !out) return perr(NPP_INVALID_ARG, "npp_proposal_create: NULL argument");
    *out = nullptr;
    if (cfg->batch < 128 || cfg->batch % 128 || cfg->batch > 65536)
        return perr(NPP_INVALID_ARG, "proposal batch must be a multiple of 128 in [128, 65536]");
    if (!(cfg->ls_min < cfg->ls_max) || !(cfg->beta1 >= 0 && cfg->beta1 < 1) || !(cfg->beta2 >= 0 && cfg->beta2 < 1) ||
        !(cfg->eps > 0))
        return perr(NPP_INVALID_ARG, "proposal config: need ls_min < ls_max, 0 <= beta < 1, eps > 0");
    cudaError_t e = cudaSetDevice(cfg->device);
    if (e != cudaSuccess) return perr(NPP_CUDA_ERROR, std::string("cudaSetDevice: ") + cudaGetErrorString(e));
    npp_proposal* P = new npp_proposal();    // all zero
    P->cfg = *cfg;
    P->B = cfg->batch;
    const size_t B = (size_t)cfg->batch;
    auto A = [&](void** p, size_t bytes) { if (e == cudaSuccess) e = cudaMalloc(p, bytes); };
    A((void**)&P->w, N_FLAT * 4); A((void**)&P->m, N_FLAT * 4); A((void**)&P->v, N_FLAT * 4); A((void**)&P->g, N_FLAT * 4);
    A((void**)&P->W1, (size_t)HID * D0 * 2); A((void**)&P->W2, (size_t)HID * HID * 2);
    A((void**)&P->W3, (size_t)D3 * HID * 2); A((void**)&P->W3f, (size_t)D3 * HID * 2);
    A((void**)&P->X, B * D0 * 2);
    A((void**)&P->H1, B * HID * 2); A((void**)&P->H2, B * HID * 2);
    A((void**)&P->dY, B * D3 * 2);
    A((void**)&P->dZ2, B * HID * 2); A((void**)&P->dZ1, B * HID * 2);
    A((void**)&P->packed, (size_t)N_PACKED * 4);
    A((void**)&P->loss, sizeof(float));
    A((void**)&P->err, sizeof(int));
    mlp_grad_splits(cfg->batch, P->splits);
    A((void**)&P->part[0], (size_t)P->splits[0] * D3 * HID * 4);
    A((void**)&P->part[1], (size_t)P->splits[1] * HID * HID * 4);
    A((void**)&P->part[2], (size_t)P->splits[2] * HID * D0 * 4);
    A((void**)&P->loss_part, B / 128 * 32 * 4);
    A((void**)&P->mask, B * 2 * 2 * sizeof(uint4));
    if (e == cudaSuccess) e = cudaMemset(P->w, 0, N_FLAT * 4);
    if (e == cudaSuccess) e = cudaMemset(P->m, 0, N_FLAT * 4);
    if (e == cudaSuccess) e = cudaMemset(P->v, 0, N_FLAT * 4);
    if (e == cudaSuccess) e = cudaMemset(P->g, 0, N_FLAT * 4);
    if (e == cudaSuccess) e = cudaMemset(P->err, 0, sizeof(int));
    // the padding inputs, the padding outputs' gradients and the padding rows
    // of the forward pass's W3 stay zero (nothing writes them)
    if (e == cudaSuccess) e = cudaMemset(P->X, 0, B * D0 * 2);
    if (e == cudaSuccess) e = cudaMemset(P->dY, 0, B * D3 * 2);
    if (e == cudaSuccess) e = cudaMemset(P->W3f, 0, (size_t)D3 * HID * 2);
    if (e != cudaSuccess) {
        npp_proposal_destroy(P);
        return perr(NPP_CUDA_ERROR, std::string("proposal allocation: ") + cudaGetErrorString(e));
    }
    const int b = cfg->batch;
    // whole K-major operand blocks; 64 x 64 boxes of the MN-major ones
    struct M { CUtensorMap* map; const void* base; int rows, cols, box; } maps[] = {
        { &P->fmaps.w1, P->W1, HID, D0, 256 }, { &P->fmaps.w2, P->W2, HID, HID, 256 },
        { &P->fmaps.w3, P->W3f, D3, HID, 256 }, { &P->fmaps.h1, P->H1, b, HID, 128 },
        { &P->fmaps.h2, P->H2, b, HID, 128 },
        { &P->bmaps.dy, P->dY, b, D3, 128 }, { &P->bmaps.w3, P->W3, D3, HID, 64 },
        { &P->bmaps.w2, P->W2, HID, HID, 64 }, { &P->bmaps.dz2, P->dZ2, b, HID, 128 },
        { &P->bmaps.dz1, P->dZ1, b, HID, 128 },
        { &P->grads.a[0], P->dY, b, D3, 64 }, { &P->grads.b[0], P->H2, b, HID, 64 },
        { &P->grads.a[1], P->dZ2, b, HID, 64 }, { &P->grads.b[1], P->H1, b, HID, 64 },
        { &P->grads.a[2], P->dZ1, b, HID, 64 }, { &P->grads.b[2], P->X, b, D0, 64 },
    };
    for (auto& mp : maps) {
        e = make_tmap_bf16(mp.map, mp.base, mp.rows, mp.cols, mp.box);
        if (e != cudaSuccess) {
            npp_proposal_destroy(P);
            return perr(NPP_CUDA_ERROR, std::string("tensor map: ") + cudaGetErrorString(e));
        }
    }
    e = refresh_bf16(P, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        npp_proposal_destroy(P);
        return perr(NPP_CUDA_ERROR, std::string("proposal init: ") + cudaGetErrorString(e));
    }
    *out = P;
    return NPP_OK;
}

npp_status npp_proposal_destroy(npp_proposal* P)
{
    if (!P) return NPP_OK;
    cudaSetDevice(P->cfg.device);
    cudaDeviceSynchronize();
    void* ptrs[] = { P->w, P->m, P->v, P->g, P->W1, P->W2, P->W3, P->W3f, P->X, P->H1, P->H2, P->dY, P->dZ2, P->dZ1,
                     P->loss, P->err, P->part[0], P->part[1], P->part[2], P->loss_part, P->mask, P->packed };
    for (void* p : ptrs) if (p) cudaFree(p);
    delete P;
    return NPP_OK;
}

npp_status npp_proposal_set_params(npp_proposal* P, const float* params_host)
{
    if (!P || !params_host) return perr(NPP_INVALID_ARG, "npp_proposal_set_params: NULL argument");
    for (int i = 0; i < N_PACKED; ++i)
        if (!std::isfinite(params_host[i])) return perr(NPP_INVALID_ARG, "proposal parameters must be finite");
    cudaSetDevice(P->cfg.device);
    float* flat = new float[N_FLAT];
    packed_to_flat(params_host, flat);
    cudaError_t e = cudaMemcpy(P->w, flat, N_FLAT * 4, cudaMemcpyHostToDevice);
    delete[] flat;
    if (e == cudaSuccess) e = cudaMemset(P->m, 0, N_FLAT * 4);
    if (e == cudaSuccess) e = cudaMemset(P->v, 0, N_FLAT * 4);
    if (e == cudaSuccess) e = refresh_bf16(P, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return perr(NPP_CUDA_ERROR, std::string("proposal set: ") + cudaGetErrorString(e));
    P->t = 0;
    return NPP_OK;
}

npp_status npp_proposal_get_params(npp_proposal* P, float* params_host)
{
    if (!P || !params_host) return perr(NPP_INVALID_ARG, "npp_proposal_get_params: NULL argument");
    cudaSetDevice(P->cfg.device);
    return read_flat(P, P->w, params_host);
}

npp_status npp_proposal_get_grads(npp_proposal* P, float* grads_host)
{
    if (!P || !grads_host) return perr(NPP_INVALID_ARG, "npp_proposal_get_grads: NULL argument");
    cudaSetDevice(P->cfg.device);
    return read_flat(P, P->g, grads_host);
}

npp_status npp_proposal_encode(const npp_handle* h, const npp_scene* scenes_dev, int32_t S, const float* obs_dev,
                               float* x_dev, void* stream)
{
    if (!h || !scenes_dev || !x_dev || S < 0) return perr(NPP_INVALID_ARG, "npp_proposal_encode: bad arguments");
    if (S == 0) return NPP_OK;
    if (!obs_dev || (reinterpret_cast<uintptr_t>(obs_dev) & 15u))
        return perr(NPP_INVALID_ARG, "npp_proposal_encode: obstacle array must be non-NULL and 16-byte aligned");
    cudaSetDevice(h->device);
    encode_kernel<<<S, ENC_THREADS, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        h->dc, scenes_dev, reinterpret_cast<const float4*>(obs_dev), x_dev);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return perr(NPP_CUDA_ERROR, std::string("encode launch: ") + cudaGetErrorString(e));
    return NPP_OK;
}

npp_status npp_proposal_forward(npp_proposal* P, const float* x_dev, int32_t n, float* mean_dev, float* std_dev,
                                void* stream)
{
    if (!P || !x_dev || !mean_dev || !std_dev) return perr(NPP_INVALID_ARG, "npp_proposal_forward: NULL argument");
    if (n < 1 || n > P->B) return perr(NPP_INVALID_ARG, "npp_proposal_forward: n outside [1, batch]");
    cudaSetDevice(P->cfg.device);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    MlpForward f = forward_args(P, x_dev, n);
    f.mean = mean_dev;
    f.sd = std_dev;
    const cudaError_t e = launch_mlp_forward(P->fmaps, f, s);
    if (e != cudaSuccess) return perr(NPP_CUDA_ERROR, std::string("proposal forward: ") + cudaGetErrorString(e));
    return NPP_OK;
}

npp_status npp_proposal_train_step(npp_proposal* P, const float* x_dev, const float* theta_dev, float lr,
                                   float* loss_dev, void* stream)
{
    if (!P || !x_dev || !theta_dev) return perr(NPP_INVALID_ARG, "npp_proposal_train_step: NULL argument");
    if (!(lr >= 0.0f) || !std::isfinite(lr)) return perr(NPP_INVALID_ARG, "learning rate must be finite and >= 0");
    cudaSetDevice(P->cfg.device);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int B = P->B;
    MlpForward f = forward_args(P, x_dev, B);
    f.theta = theta_dev;
    f.X = P->X; f.dY = P->dY; f.mask = P->mask;
    f.loss_part = P->loss_part;
    cudaError_t e = launch_mlp_forward(P->fmaps, f, s);
    if (e == cudaSuccess) {
        e = launch_mlp_backward(P->bmaps, MlpBackward{ B, P->mask, P->err }, s);
    }
    if (e == cudaSuccess) {
        MlpGrads gr = { B, { P->splits[0], P->splits[1], P->splits[2] }, { P->part[0], P->part[1], P->part[2] }, P->err };
        e = launch_mlp_grads(P->grads, gr, s);
    }
    if (e == cudaSuccess) {
        P->t += 1;
        UpdateArgs u;
        u.w = P->w; u.m = P->m; u.v = P->v; u.g = P->g;
        u.W[0] = P->W1; u.W[1] = P->W2; u.W[2] = P->W3; u.W3f = P->W3f;
        u.part[0] = P->part[2]; u.part[1] = P->part[1]; u.part[2] = P->part[0];
        u.splits[0] = P->splits[2]; u.splits[1] = P->splits[1]; u.splits[2] = P->splits[0];
        u.dz[0] = P->dZ1; u.dz[1] = P->dZ2; u.dz[2] = P->dY;
        u.batch = B;
        u.loss_part = P->loss_part;
        u.n_loss = B / 128 * 32;
        u.loss = loss_dev ? loss_dev : P->loss;
        u.adam = { lr, P->cfg.beta1, P->cfg.beta2, P->cfg.eps,
                   (float)(1.0 - std::pow((double)P->cfg.beta1, P->t)),
                   (float)(1.0 - std::pow((double)P->cfg.beta2, P->t)) };
        e = launch_dependent(update_kernel, UPD_B + UPD_W + 1, UPD_THREADS, 0, s, u);
    }
    if (e != cudaSuccess) return perr(NPP_CUDA_ERROR, std::string("proposal train step: ") + cudaGetErrorString(e));
    return NPP_OK;
}

npp_status npp_gemm_bf16(const uint16_t* A_dev, const uint16_t* B_dev, float* C_dev, int32_t M, int32_t N,
                         int32_t K, void* stream)
{
    if (!A_dev || !B_dev || !C_dev) return perr(NPP_INVALID_ARG, "npp_gemm_bf16: NULL argument");
    if (M < 128 || M % 128 || N < 128 || N % 128 || K < 64 || K % 64)
        return perr(NPP_INVALID_ARG, "npp_gemm_bf16: M, N multiples of 128 and K a multiple of 64");
    // (the tensor maps check A's and B's; the epilogue stores 16 bytes at a time)
    if (reinterpret_cast<uintptr_t>(C_dev) & 15u)
        return perr(NPP_INVALID_ARG, "npp_gemm_bf16: C must be 16-byte aligned");
    const int bn = (N % 256 == 0) ? 256 : 128, box_b = gemm_pairs(M, N) ? 128 : bn;
    CUtensorMap ta, tb;
    cudaError_t e = make_tmap_bf16(&ta, A_dev, M, K, 128);
    if (e == cudaSuccess) e = make_tmap_bf16(&tb, B_dev, N, K, box_b);
    if (e != cudaSuccess) return perr(NPP_INVALID_ARG, "npp_gemm_bf16: operands must be 16-byte aligned");
    int* err = nullptr;
    e = cudaGetSymbolAddress(reinterpret_cast<void**>(&err), g_gemm_err);
    if (e != cudaSuccess) return perr(NPP_CUDA_ERROR, std::string("gemm error flag: ") + cudaGetErrorString(e));
    e = launch_gemm(ta, tb, M, N, K, bn, box_b, C_dev, err, reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return perr(NPP_CUDA_ERROR, std::string("gemm launch: ") + cudaGetErrorString(e));
    return NPP_OK;
}

npp_status npp_gemm_status(void)
{
    int err = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&err, g_gemm_err, sizeof(int));
    if (e != cudaSuccess) return perr(NPP_CUDA_ERROR, std::string("gemm status: ") + cudaGetErrorString(e));
    if (err) {
        const int zero = 0;
        cudaMemcpyToSymbol(g_gemm_err, &zero, sizeof(int));
        return perr(NPP_DEVICE_TIMEOUT, "a GEMM pipeline wait timed out");
    }
    return NPP_OK;
}

}  // extern "C"
