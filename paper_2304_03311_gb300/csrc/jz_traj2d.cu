// jz_traj2d.cu -- the 2D instantiations of the trajectory kernel.
#include "jz_traj_kernel.cuh"

namespace jz {

// Shapes with compile-time row geometry: L = 16 and 64 (GW = 1, 4); the L =
// L_t = 64 warp teams of an even number of replicas also fix L_t and the slice step
// (four slices by two replicas at a time; 31 x 1024 trajectories 533 ms with eight
// slices of one, 527 so, 523 with the present passes).  Every other shape runs the
// generic instantiation.
TrajFn select_traj2d(const Geom& g, const LaunchShape& sh, bool hbm, bool pair)
{
    const int kind = row_kind(g, sh);
    if (!pair)
        return kind == kWhole    ? pick_traj<2, kWhole, false, 0, 0>(sh, hbm)
               : kind == kRagged ? pick_traj<2, kRagged, false, 0, 0>(sh, hbm)
                                 : pick_traj<2, kHalfTail, false, 0, 0>(sh, hbm);
    if (kind == kWhole && g.GW == 4 && g.Lt == 64 && g.nrep % 2 == 0 && sh.warp &&
        sh.team_threads == 32 && !hbm)
        return pick_traj<2, kWhole, true, 4, 1, 64, 4>(sh, hbm);
    if (kind == kWhole && g.GW == 4) return pick_traj<2, kWhole, true, 4, 1>(sh, hbm);
    if (kind == kWhole && g.GW == 1) return pick_traj<2, kWhole, true, 1, 1>(sh, hbm);
    return kind == kWhole    ? pick_traj<2, kWhole, true, 0, 0>(sh, hbm)
           : kind == kRagged ? pick_traj<2, kRagged, true, 0, 0>(sh, hbm)
                             : pick_traj<2, kHalfTail, true, 0, 0>(sh, hbm);
}

cudaError_t bounds_status_traj2d(unsigned int out[2], bool clear)
{
#ifdef JZ_BOUNDS_CHECK
    cudaError_t e = cudaMemcpyFromSymbol(out, jz_bounds_status, 2 * sizeof(unsigned int));
    if (e == cudaSuccess && clear) {
        const unsigned int z[2] = {0u, 0u};
        e = cudaMemcpyToSymbol(jz_bounds_status, z, sizeof z);
    }
    return e;
#else
    out[0] = out[1] = 0u;
    (void)clear;
    return cudaSuccess;
#endif
}

}  // namespace jz
