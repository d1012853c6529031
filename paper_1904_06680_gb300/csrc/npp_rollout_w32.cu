// Trajectory kernels for the 8-32-32-2 network.  Launch shapes (all compute
// identical values), template arguments <width, lanes per sample, warps per
// block, blocks per SM, variants, W2 quads in tensor memory>:
//   0 (default) 1 or 2 by the number of samples (rollout_wide)
//   1 four hidden units a lane, four samples a warp (64 samples per SM)
//   2 two units a lane, two samples a warp (40 samples per SM)
//   3, 4 every weight in registers <32, 16, 4, 4>
// Measured on GB300 (trajectories, us; 1 / 2 / the earlier default in
// registers): N = 40000, T = 40: 254 / 306 / 318; course N = 16384: 123 /
// 138 / 143; N = 8192: 74 / 86 / 89; N = 5003, T = 60: 91 / 75 / 85; N = 500,
// T = 40: 39 / 32 / 32.  Shape 1 issues about 285 warp instructions per step
// of four samples, 2 about 225 per step of two.
#include "npp_rollout.cuh"

namespace npp {

template <bool VAR>
static cudaError_t traj(const RolloutArgs& a, cudaStream_t s, bool wide)
{
    return wide ? launch_traj_tmem<32, 8, 4, 4, VAR, 8>(a, s) : launch_traj_tmem<32, 16, 4, 5, VAR, 8>(a, s);
}

cudaError_t launch_traj_w32(const RolloutArgs& a, cudaStream_t s, int variant)
{
    const bool wide = variant == 1 || (variant != 2 && rollout_wide(a, 8));
    if (uses_variants(a.c)) return traj<true>(a, s, wide);
    return variant >= 3 ? launch_traj<32, 16, 4, 4>(a, s) : traj<false>(a, s, wide);
}

// Trajectories with the windowed binned check (fused_kernel; template
// arguments after the trajectory kernel's: window of states, candidates
// loaded ahead per lane).  Not the library's choice at this width: on the
// course (N = 16384, T = 40, M = 2000) the default shape, 5 of 8 W2 quads in
// shared memory and windows of 8, takes 219 us per plan step against 142 in
// two kernels (1 to 4: 262, 234, 258, 242).
cudaError_t launch_fused_w32(const RolloutArgs& a, cudaStream_t s, int variant)
{
    if (uses_variants(a.c)) return launch_fused<32, 16, 4, 5, true, 5, 8, 4>(a, s);
    switch (variant) {
    case 1: return launch_fused<32, 16, 4, 4, false, 0, 16, 4>(a, s);
    case 2: return launch_fused<32, 16, 4, 4, false, 0, 8, 4>(a, s);
    case 3: return launch_fused<32, 16, 4, 3, false, 0, 16, 4>(a, s);
    case 4: return launch_fused<32, 16, 4, 5, false, 5, 16, 4>(a, s);
    default: return launch_fused<32, 16, 4, 5, false, 5, 8, 4>(a, s);
    }
}

}  // namespace npp
