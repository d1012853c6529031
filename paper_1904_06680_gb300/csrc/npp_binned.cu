// npp_binned.cu -- collision checks through per-timestep spatial binning
// (the grid build, and the check over stored trajectories; the check fused
// into the trajectory kernel lives in npp_rollout.cuh).
//
// For every horizon step h the obstacle points at time h Ts (EV frame,
// p + tau v with the brute-force kernels' arithmetic) are counting-sorted into
// a uniform grid of BIN_DIM x BIN_DIM cells centred on the vehicle.  A cell is
// wider than half the radius of the vehicle's disk around its reference point
// (plus a rounding margin), so the box around a state's vehicle overlaps at
// most 5 x 5 cells (rows of cells are contiguous runs: at most five per query,
// `cand_rows`); every point inside the vehicle lies in the box, and cell
// indices of points and of the query are clamped to the grid the same (monotone) way,
// so the queried cells hold every point that can be inside.  The per-point
// test is the brute-force one (same coefficients, same fma sequence), hence
// the collision flags are identical to checking all points.
#include <cmath>

#include <cuda_runtime.h>

#include "../../include/npp.h"
#include "npp_rollout.cuh"

using namespace npp;

namespace {

constexpr int BIN_THREADS = 1024;

// one block per horizon step
__global__ void __launch_bounds__(BIN_THREADS) bin_build_kernel(const RolloutArgs a, BinView g, int* __restrict__ cell_start,
                                                                float2* __restrict__ binned)
{
    extern __shared__ __align__(16) int cnt[];       // [BIN_NCELL]
    __shared__ int run_tot[BIN_THREADS / 32];
    const int h = blockIdx.x;
    if (h == 0 && threadIdx.x == 0) {
        // start of the plan step's minimum and sample queue
        if (a.best_key) *a.best_key = ~0ull;
        if (a.work) *a.work = 0u;
    }
    if (a.first) {
        // start of the grid check: no collision known, no step finished
        for (int i = h * BIN_THREADS + threadIdx.x; i < a.N; i += gridDim.x * BIN_THREADS) a.first[i] = 0x7fffffff;
        if (h == 0)
            for (int i = threadIdx.x; i < GRID_MAX_CHUNKS; i += BIN_THREADS) a.done[i] = 0;
    }
    const StepIn si = step_in(a);
    float s0, c0;
    sincosf(si.phi0, &s0, &c0);
    int* cs = cell_start + (size_t)h * BIN_CS_STRIDE;
    float2* out = binned + (size_t)h * a.M;
    if (a.first)
        build_step_bins<BIN_THREADS>(a.obs, a.M, si.x0, si.y0, s0, c0, (float)h * a.c.Ts, g,
                                     reinterpret_cast<unsigned short*>(cs), out, cnt, run_tot);
    else
        build_step_bins<BIN_THREADS>(a.obs, a.M, si.x0, si.y0, s0, c0, (float)h * a.c.Ts, g, cs, out, cnt, run_tot);
}

// One warp per sample over its stored states (each step's inequality rows
// recomputed from the state).  The warp checks BIN_SB consecutive steps at
// once, an 8-lane group per step: a step's candidates are the points of at
// most five cell rows, each row's cells contiguous in the sorted array; the
// group's lanes stride through each row's run, one candidate per row and
// lane loaded ahead (binned_rows_inside; longer rows one pass at a time
// after them).  The chunk's first colliding step, if any, ends the sample.  Steps
// are independent given the stored states, so checking a few past the first
// collision changes nothing; it replaces one chain of two dependent loads
// per step (cell bounds, then candidates) by one per chunk.
constexpr int BINNED_WARPS = 8;
constexpr int BIN_SB = 32 / BIN_ITEM_LANES; // steps per chunk
constexpr int BIN_GS = BIN_ITEM_LANES;      // lanes per step

template <bool POLY>
__global__ void __launch_bounds__(BINNED_WARPS * 32, 5) collide_binned_kernel(const RolloutArgs a)
{
    __shared__ float4 faces[POLY ? FP_MAX_FACES : 1];
    start_next();
    if constexpr (POLY) {
        for (int i = threadIdx.x; i < a.poly.n_faces; i += blockDim.x) faces[i] = a.poly.faces[i];
        __syncthreads();
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gid = lane / BIN_GS, gl = lane % BIN_GS;
    const BinView& g = a.bins;
    const int T = a.T, N = a.N;
    int n = blockIdx.x * BINNED_WARPS + warp;
    bool valid = n < N;
    if (a.live_in) {
        const int cnt = *a.live_n_in;
        valid = n < cnt;
        n = valid ? a.live_in[n] : 0;
    }
    // the states of this launch: all (0 .. T), or those of one chunk
    // (0 .. chunk_hi for the first, chunk_lo + 1 .. chunk_hi after it)
    const bool chunked = a.chunk_hi > 0;
    const int hs = chunked && a.chunk_lo > 0 ? a.chunk_lo + 1 : 0;
    const int he = chunked ? a.chunk_hi : T;
    unsigned long long key = ~0ull;
    bool fold = false;                       // lane 0: this warp's sample ended here (key to fold)
    unsigned ntest = 0, nstate = 0;          // this lane's candidate tests and states (measurement)
    if (valid) {
        int fh = -1;
        for (int h0 = hs; h0 <= he; h0 += BIN_SB) {
            const int h = h0 + gid;
            const bool ok = h <= he;
            const float4 z = ok ? a.traj[(size_t)h * N + n] : make_float4(0.f, 0.f, 0.f, 0.f);
            nstate += (ok && gl == 0) ? 1u : 0u;
            float sp, cp;
            sincos_r(z.z, sp, cp);
            const int* cs = g.cell_start + (size_t)(ok ? h : 0) * BIN_CS_STRIDE;
            const float2* pts = g.pts + (size_t)(ok ? h : 0) * g.M;
            const QueryBox qb = query_box(g, z.x, z.y, sp, cp);
            bool inside;
            if constexpr (POLY) {
                const PolyTest test = { a.poly, faces, z.x, z.y, cp, sp };
                inside = binned_rows_inside<1>(g, cs, pts, test, qb, ok, gl, ntest);
            } else {
                RectTest test;
                coef_rows(a.c, z.x, z.y, sp, cp, test.a, test.b);
                inside = binned_rows_inside<1>(g, cs, pts, test, qb, ok, gl, ntest);
            }
            const unsigned bal = __ballot_sync(FULL, inside);
            unsigned steps_hit = 0;
#pragma unroll
            for (int s = 0; s < BIN_SB; ++s)
                if ((bal >> (s * BIN_GS)) & ((1u << BIN_GS) - 1u)) steps_hit |= 1u << s;
            if (steps_hit) {
                fh = h0 + __ffs(steps_hit) - 1;
                break;
            }
        }
        if (lane == 0) {
            fh = discard_step(a.vfirst, n, fh);
            if (fh < 0 && he < T) {
                // collision-free so far: on to the next chunk
                a.live_out[atomicAdd(a.live_n_out, 1)] = n;
            } else {
                float J = __int_as_float(0x7f800000);
                if (fh < 0) {
                    J = a.jfree[n];
                    key = ((unsigned long long)__float_as_uint(J) << 32) | (unsigned)n;
                } else {
                    key = (1ull << 63) | ((unsigned long long)(T - fh) << 32) | (unsigned)n;
                }
                if (a.costs) a.costs[n] = J;
                if (a.first_hit) a.first_hit[n] = fh;
                fold = true;
            }
        }
    }
    if (a.counts) {
        unsigned long long t = ntest, s = nstate;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            t += __shfl_xor_sync(FULL, t, off);
            s += __shfl_xor_sync(FULL, s, off);
        }
        if (lane == 0 && valid) {
            atomicAdd(a.counts, t);
            atomicAdd(a.counts + 1, s);
        }
    }
    // each warp folds its key into the minimum on its own (no block barrier:
    // samples end at different steps); the read skips atomics that cannot win
    if (fold && a.best_key && key < *reinterpret_cast<volatile unsigned long long*>(a.best_key))
        atomicMin(a.best_key, key);
}

// ------------------------------------------------------------------ one step's grid in shared memory
// Block (x, h) checks a chunk of the samples at step h: the step's grid
// (cell starts as 16-bit offsets, 32 KB, and its M points) is copied into
// shared memory once, then every lane takes one state at a time -- its rows,
// the cell rows of its query and their runs of points, two at a time -- and a
// collision lowers the sample's first colliding step.  Blocks start in the
// order of their steps, so a sample that collided early is mostly skipped at
// later steps.  The chunk's last block to finish turns the first steps into
// costs and keys.  The candidates and the per-point test are the
// warp-per-sample kernel's, so the same flags.
//
// Why: there, a warp's four states at a time each wait for two dependent L2
// reads (cell bounds, then points; every step has its own grid, so they miss
// L1), and eight lanes repeat a state's query arithmetic.
// Bound: shared-memory bank conflicts and lanes waiting for the longest run
// of their warp.  Measured on GB300 (check after the trajectories, us,
// against the warp-per-sample kernel): course (16384 x 41 states, 2000
// points) 42 / 54, 5003 x 61 states 25 / 32, 8192 x 41 (855 points) 21 / 27,
// large (65536 x 101, 8192 points) 207 / 306; a handful of samples 11 / 7.
// (With polygons, whose test is long, lanes diverge: 316 / 134.)  The build
// writes this check's cell starts as 16 bits, and they and the points come by
// asynchronous copies, all in flight (32-bit starts through registers: plan
// steps of 2048 samples, T = 40, 41.1 us, now 39.0; 3000 x 201 states 118.0,
// now 114.7).
constexpr int GRID_THREADS = 512;
static_assert(BIN_NCELL * 2 % (16 * GRID_THREADS) == 0, "whole rounds of 16-byte copies");

// BYTES (8 or 16) from global into shared memory without a register between
template <int BYTES>
__device__ __forceinline__ void copy_async(void* dst, const void* src)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
constexpr int GRID_CS_BYTES = (BIN_NCELL + 8) * 2;

// the cells a query box overlaps
struct QueryCells {
    int ix0, ix1, iy0, iy1;
};
__device__ __forceinline__ QueryCells query_cells(const BinView& g, const QueryBox& q)
{
    QueryCells c;
    c.ix0 = bin_cell(q.x - q.rx, g);
    c.ix1 = bin_cell(q.x + q.rx, g);
    c.iy0 = bin_cell(q.y - q.ry, g);
    c.iy1 = min(bin_cell(q.y + q.ry, g), c.iy0 + BIN_MAX_ROWS - 1);
    return c;
}

__global__ void __launch_bounds__(GRID_THREADS, 2) collide_grid_kernel(const RolloutArgs a, int chunk)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned short* cs = reinterpret_cast<unsigned short*>(smem_raw);
    float2* pts = reinterpret_cast<float2*>(smem_raw + GRID_CS_BYTES);
    __shared__ int last;
    __shared__ unsigned long long red[GRID_THREADS / 32];
    const int tid = threadIdx.x, h = blockIdx.y;
    const int T = a.T, N = a.N, M = a.M;
    const int n0 = blockIdx.x * chunk, n1 = min(N, n0 + chunk);
    const BinView& g = a.bins;
    start_next();
    {
        // every copy in flight at once
        const char* src = reinterpret_cast<const char*>(g.cell_start + (size_t)h * BIN_CS_STRIDE);
#pragma unroll
        for (int i = 0; i < BIN_NCELL * 2 / 16 / GRID_THREADS; ++i) {
            const int o = (i * GRID_THREADS + tid) * 16;
            copy_async<16>(smem_raw + o, src + o);
        }
        const float2* p = g.pts + (size_t)h * M;
        for (int i = tid; i < M; i += GRID_THREADS) copy_async<8>(pts + i, p + i);
        if (tid == 0) cs[BIN_NCELL] = (unsigned short)M;
        copy_async_wait();
    }
    __syncthreads();
    for (int n = n0 + tid; n < n1; n += GRID_THREADS) {
        if (__ldcg(a.first + n) <= h) continue;
        const float4 z = a.traj[(size_t)h * N + n];
        float sp, cp;
        sincos_r(z.z, sp, cp);
        RectTest test;
        coef_rows(a.c, z.x, z.y, sp, cp, test.a, test.b);
        const QueryCells q = query_cells(g, query_box(g, z.x, z.y, sp, cp));
        bool hit = false;
        for (int iy = q.iy0; iy <= q.iy1 && !hit; ++iy) {
            const int b = cs[iy * BIN_DIM + q.ix0], e = cs[iy * BIN_DIM + q.ix1 + 1];
            // two points a pass (an odd run's last point twice)
            for (int i = b; i < e; i += 2) hit |= test(pts[i]) | test(pts[min(i + 1, e - 1)]);
        }
        if (hit) atomicMin(a.first + n, h);
    }
    // the chunk's last block: every first colliding step is in
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(a.done + blockIdx.x, 1) == T;
    __syncthreads();
    if (!last) return;
    __threadfence();
    unsigned long long best = ~0ull;
    for (int n = n0 + tid; n < n1; n += GRID_THREADS) {
        const int f = __ldcg(a.first + n);
        const int fh = discard_step(a.vfirst, n, f <= T ? f : -1);
        float J = __int_as_float(0x7f800000);
        unsigned long long key;
        if (fh < 0) {
            J = a.jfree[n];
            key = ((unsigned long long)__float_as_uint(J) << 32) | (unsigned)n;
        } else {
            key = (1ull << 63) | ((unsigned long long)(T - fh) << 32) | (unsigned)n;
        }
        if (a.costs) a.costs[n] = J;
        if (a.first_hit) a.first_hit[n] = fh;
        best = key < best ? key : best;
    }
    if (!a.best_key) return;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(FULL, best, off);
        best = o < best ? o : best;
    }
    if ((tid & 31) == 0) red[tid >> 5] = best;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < GRID_THREADS / 32; ++w) best = red[w] < best ? red[w] : best;
        atomicMin(a.best_key, best);
    }
}

// The grid check's work counters, from its results: a sample's states up to
// its first collision (all without one) and the points in the cells their
// boxes overlap.  The check itself cannot count: which states of a collided
// sample it still meets depends on the order in which the steps' blocks run.
// Timed plan steps only, after the last event.
// (One pair of global atomics a block: one a warp took 30 us on the course.)
constexpr int COUNT_THREADS = 256;
constexpr int COUNT_SAMPLES = 4 * COUNT_THREADS;
__global__ void __launch_bounds__(COUNT_THREADS) count_grid_kernel(const RolloutArgs a)
{
    __shared__ unsigned sum[2];
    const int h = blockIdx.y, n0 = blockIdx.x * COUNT_SAMPLES, n1 = min(a.N, n0 + COUNT_SAMPLES);
    const BinView& g = a.bins;
    const unsigned short* cs = reinterpret_cast<const unsigned short*>(g.cell_start + (size_t)h * BIN_CS_STRIDE);
    if (threadIdx.x < 2) sum[threadIdx.x] = 0u;
    __syncthreads();
    unsigned tests = 0, states = 0;
    for (int n = n0 + threadIdx.x; n < n1; n += COUNT_THREADS) {
        if (h > a.first[n]) continue;
        const float4 z = a.traj[(size_t)h * a.N + n];
        float sp, cp;
        sincos_r(z.z, sp, cp);
        const QueryCells q = query_cells(g, query_box(g, z.x, z.y, sp, cp));
        for (int iy = q.iy0; iy <= q.iy1; ++iy) tests += cs[iy * BIN_DIM + q.ix1 + 1] - cs[iy * BIN_DIM + q.ix0];
        ++states;
    }
    tests = __reduce_add_sync(FULL, tests);
    states = __reduce_add_sync(FULL, states);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&sum[0], tests);
        atomicAdd(&sum[1], states);
    }
    __syncthreads();
    if (threadIdx.x < 2 && sum[1]) atomicAdd(a.counts + threadIdx.x, (unsigned long long)sum[threadIdx.x]);
}

}  // namespace

namespace npp {

// bytes of the per-step grids: (T+1) cell-start tables and (T+1) x M points
size_t binned_workspace_bytes(int max_T, int max_M)
{
    return (size_t)(max_T + 1) * BIN_CS_STRIDE * sizeof(int) + (size_t)(max_T + 1) * max_M * sizeof(float2);
}

// the grids of geometry g into the workspace (fills a.bins)
static cudaError_t build_grids(RolloutArgs& a, BinView g, void* workspace, cudaStream_t s)
{
    int* cell_start = static_cast<int*>(workspace);
    float2* binned = reinterpret_cast<float2*>(cell_start + (size_t)(a.T + 1) * BIN_CS_STRIDE);
    g.cell_start = cell_start;
    g.pts = binned;
    g.M = a.M;
    const int smem = BIN_NCELL * (int)sizeof(int);
    cudaError_t e = ensure_smem(bin_build_kernel, smem);
    if (e != cudaSuccess) return e;
    bin_build_kernel<<<a.T + 1, BIN_THREADS, smem, s>>>(a, g, cell_start, binned);
    e = cudaGetLastError();
    if (e == cudaSuccess) a.bins = g;
    return e;
}

cudaError_t build_bins(RolloutArgs& a, float half_len, float half_wid, float c_off, void* workspace, cudaStream_t s)
{
    return build_grids(a, make_bin_grid(half_len, half_wid, c_off), workspace, s);
}

cudaError_t build_bins_poly(RolloutArgs& a, double radius, const double box[4], void* workspace, cudaStream_t s)
{
    return build_grids(a, make_bin_grid_box(radius, box), workspace, s);
}

// points that leave two blocks per SM (the offsets are 16-bit)
int collide_grid_points() { return (100 * 1024 - GRID_CS_BYTES) / 8; }

cudaError_t launch_collide_grid(const RolloutArgs& a, cudaStream_t s)
{
    // chunks of the samples: (chunk, step) blocks about three per SM, each of
    // two states a thread at most -- fewer blocks would leave SMs idle, more
    // would copy the grids oftener, and longer chunks leave the last blocks
    // running alone (four or ten states a thread: 20000 x 101 states 227 us
    // the plan step, now 185; 40000 x 61 242, now 217; one: 8192 x 41 54, not
    // 52)
    const int want = max(1, 3 * a.sm_count / (a.T + 1));
    const auto whole = [](int n) { return (n + GRID_THREADS - 1) / GRID_THREADS * GRID_THREADS; };
    const int chunk = max(min(whole((a.N + want - 1) / want), 2 * GRID_THREADS),
                          whole((a.N + GRID_MAX_CHUNKS - 1) / GRID_MAX_CHUNKS));
    const dim3 grid((a.N + chunk - 1) / chunk, a.T + 1);
    const int smem = GRID_CS_BYTES + a.M * (int)sizeof(float2);
    // the setting belongs to the kernel and the device, whichever thread or
    // handle launches: always the largest size, never this call's (another
    // thread's larger launch between this and its own setting would fail)
    const cudaError_t e = ensure_smem(collide_grid_kernel, GRID_CS_BYTES + collide_grid_points() * (int)sizeof(float2));
    if (e != cudaSuccess) return e;
    collide_grid_kernel<<<grid, GRID_THREADS, smem, s>>>(a, chunk);
    return cudaGetLastError();
}

cudaError_t launch_count_grid(const RolloutArgs& a, cudaStream_t s)
{
    count_grid_kernel<<<dim3((a.N + COUNT_SAMPLES - 1) / COUNT_SAMPLES, a.T + 1), COUNT_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_collide_binned(const RolloutArgs& a, cudaStream_t s)
{
    const int grid = (a.N + BINNED_WARPS - 1) / BINNED_WARPS;
    if (a.poly.n_faces > 0) collide_binned_kernel<true><<<grid, BINNED_WARPS * 32, 0, s>>>(a);
    else collide_binned_kernel<false><<<grid, BINNED_WARPS * 32, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace npp
