// npp_poly.cu -- the collision check of a general footprint (Sect. II-D:
// the EV as an arbitrarily refined polytope, convex or non-convex, checked
// by the linear inequalities A(phi)(p - [x, y]) < b(phi)): the union of
// convex pieces given as half-planes in the vehicle's frame, over every point
// of a step (npp_binned.cu checks it over the per-step grids).
#include <cmath>

#include <cuda_runtime.h>

#include "../../include/npp.h"
#include "npp_rollout.cuh"

using namespace npp;

namespace {

constexpr int POLY_WARPS = 8;

// Polygon footprint check against every point (the binned one is
// collide_binned_kernel's, with the same per-point test): one warp per sample
// over the stored states, h in order; the lanes stride through the step's
// points and a ballot ends the sample at its first colliding step.  Faces are
// staged in shared memory (uniform reads).
__global__ void __launch_bounds__(POLY_WARPS * 32) collide_poly_kernel(const RolloutArgs a)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ float4 faces[FP_MAX_FACES];
    const int nf = a.poly.n_faces;
    for (int i = threadIdx.x; i < nf; i += blockDim.x) faces[i] = a.poly.faces[i];
    __syncthreads();
    const BinView& g = a.bins;
    const int T = a.T, N = a.N, M = a.M;
    const int n = blockIdx.x * POLY_WARPS + warp;
    unsigned long long key = ~0ull;
    if (n < N) {
        int fh = -1;
        float4 nz = a.traj[n];
        for (int h = 0; h <= T; ++h) {
            const float4 z = nz;
            if (h < T) nz = a.traj[(size_t)(h + 1) * N + n];
            float sp, cp;
            sincos_r(z.z, sp, cp);
            const float2* pts = g.pts + (size_t)h * M;
            bool hit = false;
            for (int base = 0; base < M && !hit; base += 32) {
                const int k = base + lane;
                bool inside = false;
                if (k < M)
                    inside = poly_inside(a.poly, faces, pts[k], z.x, z.y, cp, sp);
                hit = __any_sync(FULL, inside);
            }
            if (hit) { fh = h; break; }
        }
        if (lane == 0) {
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
    }
    // each warp folds its key into the minimum on its own (no block barrier:
    // samples end at different steps); the read skips atomics that cannot win
    if (lane == 0 && n < N && a.best_key && key < *reinterpret_cast<volatile unsigned long long*>(a.best_key))
        atomicMin(a.best_key, key);
}

}  // namespace

namespace npp {

cudaError_t launch_collide_poly(const RolloutArgs& a, cudaStream_t s)
{
    collide_poly_kernel<<<(a.N + POLY_WARPS - 1) / POLY_WARPS, POLY_WARPS * 32, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace npp
