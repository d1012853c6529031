// Trajectory kernels for the 8-64-64-2 network.  Launch shapes (all compute
// identical values), template arguments <width, lanes per sample, warps per
// block, blocks per SM, variants, W2 quads in tensor memory, in shared
// memory>:
//   0 (default) 1 from 16384 samples on, else 2
//   1 four hidden units a lane, two samples a warp, half of W2 in shared
//     memory (24 samples per SM)
//   2 two units a lane, one sample a warp, W2 in tensor memory (16 per SM)
//   3, 4 the last 8 of each lane's 16 W2 quads in shared memory, the rest in
//     registers <64, 32, 1, 16, false, 8>
// Measured on GB300 (trajectories, us; 1 / 2 / 3): N = 65536, T = 100: 2590 /
// 2782 / 3321; N = 2000, T = 50: 104 / 78 / 96.  A wave of shape 1 holds 3648
// samples and takes 1.4 times a wave of 2 (2432 samples), so rounding to
// waves decides below a few of them.
#include "npp_rollout.cuh"

namespace npp {

template <bool VAR>
static cudaError_t traj(const RolloutArgs& a, cudaStream_t s, bool wide)
{
    return wide ? launch_traj_tmem<64, 16, 4, 3, VAR, 8, 8>(a, s) : launch_traj_tmem<64, 32, 4, 4, VAR, 16>(a, s);
}

cudaError_t launch_traj_w64(const RolloutArgs& a, cudaStream_t s, int variant)
{
    const bool wide = variant == 1 || (variant != 2 && a.N >= 16384);
    if (uses_variants(a.c)) return traj<true>(a, s, wide);
    return variant >= 3 ? launch_traj<64, 32, 1, 16, false, 8>(a, s) : traj<false>(a, s, wide);
}

// Trajectories with the windowed binned check (template arguments after the
// trajectory kernel's: window of states, candidates loaded ahead per lane).
// Default: 24 warps per SM in one block, 10 of 16 W2 quads in tensor memory
// and 6 in shared memory, windows of 8 states; below 160 samples per SM
// four-warp blocks, 16 warps per SM, with all of W2 in tensor memory: a
// sample runs through faster, which counts until the queue is long.
// Measured on GB300 (us): N = 65536, T = 100, M = 8192: 16 warps per SM 2018, 20
// (12 quads) 1993, 24 1976; shape 3, the earlier default in registers and
// shared memory (one sample per block), 2458; two samples a warp, 12 warps,
// 2350.  Plan steps with 24 / 16 warps, T = 50, M = 4000: N = 2432 125 / 102,
// 4800 173 / 154, 9000 244 / 235, 24000 529 / 528, 48000 992 / 1001.
// (Windows of 4 states take 3 % less, but the library's work counters are
// defined by windows of 8.)
template <bool VAR>
static cudaError_t fused(const RolloutArgs& a, cudaStream_t s, bool full)
{
    return full ? launch_fused_tmem<64, 32, 24, 1, VAR, 10, 6, 8, 4>(a, s)
                : launch_fused_tmem<64, 32, 4, 4, VAR, 16, 0, 8, 4>(a, s);
}

cudaError_t launch_fused_w64(const RolloutArgs& a, cudaStream_t s, int variant)
{
    const bool full = variant == 1 || (variant != 2 && a.N >= 160 * a.sm_count);
    if (uses_variants(a.c)) return fused<true>(a, s, full);
    return variant >= 3 ? launch_fused<64, 32, 1, 16, false, 12, 8, 4>(a, s) : fused<false>(a, s, full);
}

}  // namespace npp
