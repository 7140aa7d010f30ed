// jz_kernels.cu -- the FP64 estimator of one job, and the launch of the
// trajectory kernel (jz_traj_kernel.cuh).
#include <cstdint>

#include "jz_traj_kernel.cuh"

namespace jz {

// ---------------------------------------------------------------- estimator --
// One CTA: ln <e^-W> with W_i = scale * w_int[i] as a max-shifted log-sum-exp
// per jackknife block, then the full and leave-one-block-out estimates
// (Appendix A, eq. Jarzynski_theorem; blocked jackknife).
// out[0] = ln <e^-W>, out[1] = Delta S_2, out[2] = jackknife error.
constexpr int kMaxJackBlocks = 64;

__global__ void __launch_bounds__(1024)
estimator_kernel(const long long* __restrict__ w_int, int n, double scale, int direction,
                 int n_blocks, double* __restrict__ out)
{
    __shared__ double s_max[kMaxJackBlocks], s_sum[kMaxJackBlocks];
    __shared__ int s_lo[kMaxJackBlocks + 1];
    __shared__ double s_theta[kMaxJackBlocks + 1];
    const int B = n_blocks;
    const int size = n / B;
    if (threadIdx.x <= B) s_lo[threadIdx.x] = threadIdx.x == B ? n : threadIdx.x * size;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_warps = blockDim.x >> 5;
    for (int b = warp; b < B; b += n_warps) {
        const int lo = s_lo[b], hi = s_lo[b + 1];
        double m = -INFINITY;
        for (int i = lo + lane; i < hi; i += 32) m = fmax(m, -scale * (double)w_int[i]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
        double acc = 0.0;
        for (int i = lo + lane; i < hi; i += 32) acc += exp(-scale * (double)w_int[i] - m);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
        if (lane == 0) { s_max[b] = m; s_sum[b] = acc; }
    }
    __syncthreads();
    estimator_finish(s_max, s_sum, s_lo, B, n, direction, s_theta, out);
}

// ------------------------------------------------------------ host launchers --
size_t traj_smem_bytes(const Geom& g) { return (size_t)2 * g.NR * g.GW * sizeof(uint32_t); }

bool traj_pairs(const Geom& g, int teams, bool hbm)
{
    return (hbm ? 0 : traj_smem_bytes(g) * teams) + kPairReserve <= kMaxDynSmem;
}

static TrajFn select_traj(int D, const Geom& g, const LaunchShape& sh, bool hbm, bool pair)
{
    return D == 2 ? select_traj2d(g, sh, hbm, pair) : select_traj3d(g, sh, hbm, pair);
}

// Lets kern take up to the per-CTA maximum of dynamic shared memory.  The
// attribute is raised once to that maximum, never lowered, so that launches
// and occupancy queries of the same kernel from several host threads with
// different lattice sizes cannot narrow it under one another.
static cudaError_t open_smem(TrajFn kern)
{
    cudaFuncAttributes fa;
    int dev = 0, optin = 0;
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const int max_dyn = optin - (int)fa.sharedSizeBytes;
    if (fa.maxDynamicSharedSizeBytes >= max_dyn) return cudaSuccess;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn);
}

static size_t dyn_smem(const Geom& g, const LaunchShape& sh, bool hbm, bool pair)
{
    return (hbm ? 0 : traj_smem_bytes(g) * sh.teams) + (pair ? kPairTable * sizeof(uint2) : 0);
}

cudaError_t launch_traj(int D, const Geom& g, const PhiloxKeys& K, const JobDesc* jobs,
                        int n_jobs, long long n_cta, const LaunchShape& sh, bool never,
                        cudaStream_t st, uint32_t* gS)
{
    const bool hbm = gS != nullptr;
    const bool pair = !never && traj_pairs(g, sh.teams, hbm);
    const TrajFn kern = select_traj(D, g, sh, hbm, pair);
    const cudaError_t e = open_smem(kern);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)n_cta, sh.cta_threads, dyn_smem(g, sh, hbm, pair), st>>>(g, K, jobs, n_jobs,
                                                                             sh, gS);
    return cudaGetLastError();
}

cudaError_t traj_occupancy(int D, const Geom& g, const LaunchShape& sh, int* ctas_per_sm)
{
    const bool pair = traj_pairs(g, sh.teams, false);
    const TrajFn kern = select_traj(D, g, sh, false, pair);
    const cudaError_t e = open_smem(kern);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, kern, sh.cta_threads,
                                                         dyn_smem(g, sh, false, pair));
}

cudaError_t launch_estimator(const long long* w_int, int n, double scale, int direction,
                             int n_blocks, double* out, cudaStream_t st)
{
    estimator_kernel<<<1, 1024, 0, st>>>(w_int, n, scale, direction, n_blocks, out);
    return cudaGetLastError();
}

}  // namespace jz
