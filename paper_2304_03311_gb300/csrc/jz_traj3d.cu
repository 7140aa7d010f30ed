// jz_traj3d.cu -- the 3D instantiations of the trajectory kernel.
#include "jz_traj_kernel.cuh"

namespace jz {

// L = 16 (GW = 1, L_y = 16) has compile-time row geometry; every other shape
// runs the generic instantiation.
TrajFn select_traj3d(const Geom& g, const LaunchShape& sh, bool hbm, bool pair)
{
    const int kind = row_kind(g, sh);
    if (!pair)
        return kind == kWhole   ? pick_traj<3, kWhole, false, 0, 0>(sh, hbm)
               : kind == kRagged ? pick_traj<3, kRagged, false, 0, 0>(sh, hbm)
                                 : pick_traj<3, kHalfTail, false, 0, 0>(sh, hbm);
    if (kind == kWhole && g.GW == 1 && g.Ly == 16) return pick_traj<3, kWhole, true, 1, 16>(sh, hbm);
    return kind == kWhole   ? pick_traj<3, kWhole, true, 0, 0>(sh, hbm)
           : kind == kRagged ? pick_traj<3, kRagged, true, 0, 0>(sh, hbm)
                             : pick_traj<3, kHalfTail, true, 0, 0>(sh, hbm);
}

cudaError_t bounds_status_traj3d(unsigned int out[2], bool clear)
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
