// Trajectory kernels for the 8-16-16-2 network.  Launch shapes (all compute
// identical values), template arguments <width, lanes per sample, warps per
// block, blocks per SM, variants, W2 quads in tensor memory>:
//   0 (default) 1 or 2 by the number of samples (rollout_wide)
//   1 four hidden units a lane, eight samples a warp: fewer instructions per
//     sample, so the faster one where samples fill the SMs
//   2 two units a lane, four samples a warp: more warps from the same
//     samples and a shorter chain per step, so the faster one below
//   1's samples in 20-warp blocks (LEAN) where they fill 20 warps per SM but
//     not 16 (N in 16 .. 20 x 8 x SMs), a second wave otherwise: N = 20480,
//     T = 200: 225 -> 190; N = 24320, T = 40: 81 -> 71.  In one wave of 16
//     or in several the 16-warp shape is the faster (16384 samples, T = 40:
//     56 / 61; 30000: 91 / 113).
//   3, 4 every weight in registers <16, 8, 4, 4>
// Measured on GB300 (trajectories, us; 1 / 2 / the earlier default in
// registers): road N = 20480, T = 200: 223 / 248 / 280; course N = 16384,
// T = 40: 58 / 70 / 72; N = 4096: 38 / 37 / 42; N = 256, T = 20: 20 / 18 / 20.
#include "npp_rollout.cuh"

namespace npp {

template <bool VAR>
static cudaError_t traj(const RolloutArgs& a, cudaStream_t s, bool wide)
{
    // samples that 16 warps per SM take in a wave and a bit, and 20 in one
    const int per = 8 * a.sm_count;
    if (wide && a.N > 16 * per && a.N <= 20 * per) return launch_traj_tmem<16, 4, 20, 1, VAR, 4, 0, true>(a, s);
    return wide ? launch_traj_tmem<16, 4, 4, 4, VAR, 4>(a, s) : launch_traj_tmem<16, 8, 4, 6, VAR, 4>(a, s);
}

cudaError_t launch_traj_w16(const RolloutArgs& a, cudaStream_t s, int variant)
{
    const bool wide = variant == 1 || (variant != 2 && rollout_wide(a, 16));
    if (uses_variants(a.c)) return traj<true>(a, s, wide);
    return variant >= 3 ? launch_traj<16, 8, 4, 4>(a, s) : traj<false>(a, s, wide);
}

// Trajectories with the windowed binned check (fused_kernel; template
// arguments after the trajectory kernel's: window of states, candidates
// loaded ahead per lane).  Not the library's choice at this width: 182 us per
// plan step of the course (N = 16384, T = 40, M = 2000) against 84 in two
// kernels (2: 163, 3: 189)
cudaError_t launch_fused_w16(const RolloutArgs& a, cudaStream_t s, int variant)
{
    if (uses_variants(a.c)) return launch_fused<16, 8, 4, 4, true, 0, 16, 4>(a, s);
    switch (variant) {
    case 2: return launch_fused<16, 8, 4, 4, false, 0, 8, 4>(a, s);
    case 3: return launch_fused<16, 8, 4, 4, false, 0, 16, 2>(a, s);
    default: return launch_fused<16, 8, 4, 4, false, 0, 16, 4>(a, s);
    }
}

}  // namespace npp
