// Collision kernels with all obstacle points resident in shared memory.
// Variants compute the same values: 0 block-balanced (16 warps, one block per
// SM, items of up to 128 samples); 1 block-balanced with 8 warps and two
// blocks per SM; 2 warp-owned items of 8 samples pulled from a queue; 3 / 4
// items of 8 samples on 4 / 2 point slices, two / four items per 8-warp
// block sharing one staged copy of the points (two blocks per SM).  Besides
// them, for a few points, the state-parallel kernel (one lane per state).
#include "npp_rollout.cuh"

namespace npp {

// ------------------------------------------------------------------ a few points: one lane per state
// A warp takes S = 32 / P samples at P consecutive steps, one state per lane,
// round by round; every lane runs through all the points (EV-frame pairs in
// shared memory, read by all lanes at once) with the brute-force per-point
// test, and a sample ends with the first colliding step of its round.
// Steps are independent given the stored states, so checking up to P - 1
// past the first collision changes nothing.
//
// The kernels that spread a step's points over the lanes leave most lanes
// idle when the points are few (20 points are 10 pairs) and pay a warp vote
// per sample and step: about 270 us for N = 20480, T = 200, M = 20.  Here
// every lane works whatever the number of points, about 45 + 11 M / 2
// instructions per state with no vote but one per round: about 40 us there
// (the climb of 15 such rounds 8.24 -> 4.85 ms).
// Bound: FP32 issue.
constexpr int STATES_WARPS = 8;

template <int P>
__global__ void __launch_bounds__(STATES_WARPS * 32) collide_states_kernel(const RolloutArgs a)
{
    constexpr int S = 32 / P;
    extern __shared__ __align__(16) float4 pairs[];              // XY_q at 2 q, V_q at 2 q + 1
    const int tid = threadIdx.x, lane = tid & 31;
    const int T = a.T, N = a.N, npairs = (a.M + 1) / 2;
    start_next();
    {
        const StepIn si = step_in(a);
        float s0, c0;
        sincosf(si.phi0, &s0, &c0);
        for (int q = tid; q < npairs; q += STATES_WARPS * 32) {
            float px[2], py[2], vx[2], vy[2];
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const int j = 2 * q + o;
                px[o] = 1e15f; py[o] = 1e15f; vx[o] = 0.f; vy[o] = 0.f;
                if (j < a.M) ev_point(a.obs[j], si.x0, si.y0, s0, c0, px[o], py[o], vx[o], vy[o]);
            }
            pairs[2 * q] = make_float4(px[0], px[1], py[0], py[1]);
            pairs[2 * q + 1] = make_float4(vx[0], vx[1], vy[0], vy[1]);
        }
    }
    __syncthreads();
    wait_for_previous();                                         // the trajectories
    const int sl = lane % S, ph = lane / S;                      // sample and step of this lane
    const int n = (blockIdx.x * STATES_WARPS + (tid >> 5)) * S + sl;
    const bool valid = n < N;
    unsigned mine = 0;                                           // the lanes of this lane's sample
#pragma unroll
    for (int p = 0; p < P; ++p) mine |= 1u << (p * S);
    mine <<= sl;
    bool alive = valid;
    int fh = -1;
    float4 nz = make_float4(0.f, 0.f, 0.f, 0.f);
    if (alive && ph <= T) nz = a.traj[(size_t)ph * N + n];
    for (int h0 = 0; h0 <= T; h0 += P) {
        const int h = h0 + ph;
        const float4 z = nz;
        if (alive && h + P <= T) nz = a.traj[(size_t)(h + P) * N + n];
        float4 ca;
        float2 cb;
        rows_of_state(a.c, z, ca, cb);
        const unsigned long long A = pk(ca.x, ca.x), B = pk(ca.y, ca.y), NC = pk(ca.z, ca.z);
        const unsigned long long D = pk(ca.w, ca.w), E = pk(cb.x, cb.x), NF = pk(cb.y, cb.y);
        const float tau = (float)h * a.c.Ts;
        const unsigned long long TT = pk(tau, tau);
        unsigned long long acc = 0ull;
#pragma unroll 4
        for (int q = 0; q < npairs; ++q) {
            const float4 xy = pairs[2 * q], vv = pairs[2 * q + 1];
            const unsigned long long PX = fma2(TT, pk(vv.x, vv.y), pk(xy.x, xy.y));
            const unsigned long long PY = fma2(TT, pk(vv.z, vv.w), pk(xy.z, xy.w));
            const unsigned long long xi = fma2(A, PX, fma2(B, PY, NC));
            const unsigned long long et = fma2(D, PX, fma2(E, PY, NF));
            acc |= ~(xi | et);
        }
        const bool inside = ((((unsigned)acc) | (unsigned)(acc >> 32)) >> 30) & 1u;
        const unsigned hits = __ballot_sync(FULL, alive && h <= T && inside) & mine;
        if (hits) {
            fh = h0 + (__ffs(hits) - 1) / S;
            alive = false;
        }
        if (!__any_sync(FULL, alive)) break;
    }
    unsigned long long key = ~0ull;
    if (valid && ph == 0) {
        fh = discard_step(a.vfirst, n, fh);
        float J = __int_as_float(0x7f800000);
        if (fh < 0) {
            J = a.jfree[n];
            key = ((unsigned long long)__float_as_uint(J) << 32) | (unsigned)n;
        } else {
            key = (1ull << 63) | ((unsigned long long)(T - fh) << 32) | (unsigned)n;
        }
        if (a.costs) a.costs[n] = J;
        if (a.first_hit) a.first_hit[n] = fh;
    }
    if (!a.best_key) return;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(FULL, key, off);
        key = o < key ? o : key;
    }
    // the read skips atomics that cannot win
    if (lane == 0 && key < *reinterpret_cast<volatile unsigned long long*>(a.best_key)) atomicMin(a.best_key, key);
}

template <int P>
static cudaError_t launch_states(const RolloutArgs& a, cudaStream_t s)
{
    constexpr int per_block = STATES_WARPS * (32 / P);
    return launch_dependent(collide_states_kernel<P>, (a.N + per_block - 1) / per_block, STATES_WARPS * 32,
                            (size_t)((a.M + 1) / 2 * 32), s, a);
}

// One sample per warp, 32 steps a round, except for many samples with few
// points and steps: there the state reads count, and at two samples per warp
// they fill their 32-byte sectors.  Over long horizons the more and shorter
// warps of one sample each win: they fill the SMs as the trajectories' blocks
// leave, without a nearly empty last wave.  Measured on GB300 (plan step, P =
// 4, 8, 16, 32): N = 20480, T = 60, M = 20: 126, 123, 122, 124 us; N = 2048,
// T = 40, M = 128: 66, 52, 44, 43 us; later, P = 16, 32, M = 20: N = 20480, T = 60
// 86, 89, T = 200 226, 223; N = 8192, T = 200 126, 121; N = 40960, T = 200 429,
// 431 (many waves: the two differ by less than 1 % there).
cudaError_t launch_collide_states(const RolloutArgs& a, cudaStream_t s)
{
    return a.N >= 8192 && a.M < 64 && a.T < 128 ? launch_states<16>(a, s) : launch_states<32>(a, s);
}

using CollideResident = CollideBlockKernel<16, 128>;

cudaError_t launch_collide_resident(const RolloutArgs& a, cudaStream_t s, int variant)
{
    switch (variant) {
    case 0: return launch_collide_block<16, 128, 1>(a, s);
    case 1: return launch_collide_block<8, 64, 2>(a, s);
    case 2: return launch_collide_warp<8, 2>(a, s);
    case 3: return launch_collide_slice<4, 2, 2>(a, s);
    default: return launch_collide_slice<2, 2, 4>(a, s);
    }
}

int collide_resident_blocks_per_sm(int M, int variant)
{
    switch (variant) {
    case 0: return collide_block_blocks_per_sm<16, 128, 1>(M);
    case 1: return collide_block_blocks_per_sm<8, 64, 2>(M);
    case 2: return collide_warp_blocks_per_sm<8, 2>(M);
    case 3: return collide_slice_blocks_per_sm<4, 2, 2>(M);
    default: return collide_slice_blocks_per_sm<2, 2, 4>(M);
    }
}

cudaError_t launch_collide_global(const RolloutArgs& a, cudaStream_t s)
{
    return launch_collide_slice_global<4, 4>(a, s);
}

int collide_global_blocks_per_sm()
{
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, collide_slice_kernel<4, 4, true>, 128,
                                                  CollideSliceKernel<4>::fixed_bytes());
    return nb > 0 ? nb : 1;
}

// points whose pair blocks fit beside the largest fixed part (and the
// staging barrier, static shared memory)
int collide_max_points(int smem_limit)
{
    return 64 * ((smem_limit - CollideResident::fixed_bytes() - 16) / 1024);
}

}  // namespace npp
