// jz_kernels.cu -- the FP64 estimator of one job, and the launch of the
// trajectory kernel (jz_traj_kernel.cuh).
#include <cstdint>

#include "jz_host.h"
#include "jz_traj_kernel.cuh"

namespace jz {

// ---------------------------------------------------------------- estimator --
// One CTA: ln <e^-W> with W_i = scale * w_int[i] as a max-shifted log-sum-exp
// per jackknife block, then the full and leave-one-block-out estimates
// (Appendix A, eq. Jarzynski_theorem; blocked jackknife).
// out[0] = ln <e^-W>, out[1] = Delta S_2, out[2] = jackknife error.
constexpr int kMaxJackBlocks = 64;
constexpr int kEstThreads = 160, kEstOneCta = 1024;
static_assert(kEstThreads >= kEstFinish && kEstOneCta >= kEstFinish, "");

__global__ void __launch_bounds__(kEstOneCta)
estimator_kernel(const long long* __restrict__ w_int, int n, double scale, int direction,
                 int n_blocks, double* __restrict__ out)
{
    __shared__ double s_max[kMaxJackBlocks], s_sum[kMaxJackBlocks];
    __shared__ int s_lo[kMaxJackBlocks + 1];
    __shared__ double s_theta[kMaxJackBlocks + 1], s_exp[2 * kMaxJackBlocks];
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
    estimator_finish(s_max, s_sum, s_lo, B, n, direction, s_theta, s_exp, out);
}

// The same estimate by a grid of B x C CTAs: CTA (b, c) reduces chunk c of
// jackknife block b to its maximum and shifted sum in part[], and the last
// CTA to finish (counted in *done, which it sets back to 0) joins the chunks
// and forms the estimates.
//
// What bounds it: FP64 exponentials, about 20 FP64 operations each, at two FP64
// lanes per clock and SM: 16384 of them take one SM 85 us and 96 SMs 1 us; then the
// finish on one CTA and the call.  A chunk holds a value per thread and up to as many
// again (the chunk count rounds down): 16384 values, B = 32, are 96 CTAs of 170 or 171
// values on 160 threads.  Whole call: 153 us on one CTA -> 25 us (kernel about 15 us).
__global__ void __launch_bounds__(kEstThreads)
estimator_grid_kernel(const long long* __restrict__ w_int, int n, double scale, int direction,
                      int B, int C, double2* part, unsigned int* done, double* __restrict__ out)
{
    __shared__ double s_max[kMaxJackBlocks], s_sum[kMaxJackBlocks];
    __shared__ int s_lo[kMaxJackBlocks + 1];
    __shared__ double s_theta[kMaxJackBlocks + 1], s_exp[2 * kMaxJackBlocks];
    __shared__ double s_red[2][kEstThreads / 32], s_part[kEstMaxCtas];
    __shared__ bool s_last;
    const int t = (int)threadIdx.x, warp = t >> 5, lane = t & 31;
    const int size = n / B;
    const int b = (int)blockIdx.x / C, c = (int)blockIdx.x - b * C;
    const int len = b == B - 1 ? n - b * size : size;
    const int lo = b * size + (int)((long long)len * c / C);
    const int hi = b * size + (int)((long long)len * (c + 1) / C);
    auto reduce = [&](double v, bool mx, double* red) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double x = __shfl_xor_sync(0xFFFFFFFFu, v, o);
            v = mx ? fmax(v, x) : v + x;
        }
        if (lane == 0) red[warp] = v;
        __syncthreads();
        v = red[0];
#pragma unroll
        for (int i = 1; i < kEstThreads / 32; ++i) v = mx ? fmax(v, red[i]) : v + red[i];
        return v;
    };
    const int i0 = lo + t;
    const double x0 = i0 < hi ? -scale * (double)w_int[i0] : -INFINITY;
    double m = x0;
    for (int i = i0 + kEstThreads; i < hi; i += kEstThreads)
        m = fmax(m, -scale * (double)w_int[i]);
    m = reduce(m, true, s_red[0]);
    double acc = i0 < hi ? exp(x0 - m) : 0.0;
    for (int i = i0 + kEstThreads; i < hi; i += kEstThreads)
        acc += exp(-scale * (double)w_int[i] - m);
    acc = reduce(acc, false, s_red[1]);
    if (t == 0) {
        part[blockIdx.x] = make_double2(m, acc);
        __threadfence();
        s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (t <= B) s_lo[t] = t == B ? n : t * size;
    if (t < B) {
        double M = -INFINITY;
        for (int k = 0; k < C; ++k) M = fmax(M, __ldcg(&part[t * C + k].x));
        s_max[t] = M;
    }
    __syncthreads();
    for (int i = t; i < B * C; i += kEstThreads) {
        const double2 p = __ldcg(&part[i]);
        const double M = s_max[i / C];
        s_part[i] = p.x == M ? p.y : p.y * exp(p.x - M);
    }
    __syncthreads();
    if (t < B) {
        double S = 0.0;
        for (int k = 0; k < C; ++k) S += s_part[t * C + k];
        s_sum[t] = S;
    }
    if (t == 0) *done = 0u;
    __syncthreads();
    estimator_finish(s_max, s_sum, s_lo, B, n, direction, s_theta, s_exp, out);
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
    // The one-row path counts thresholds itself, for any couplings, and lives in
    // the instantiation with the table (1000 trajectories of 200 sweeps at beta = 3:
    // 0.15 ms, 0.27 ms by the general counting kernel).
    const bool rows = D == 2 && g.Lh == 8 && sh.warp && one_row_team(g, sh);
    const bool pair = (!never || rows) && traj_pairs(g, sh.teams, hbm);
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
    estimator_kernel<<<1, kEstOneCta, 0, st>>>(w_int, n, scale, direction, n_blocks, out);
    return cudaGetLastError();
}

// Chunks per jackknife block: as many as hold a value per thread, up to kEstMaxCtas
// CTAs.
cudaError_t launch_estimator_grid(const long long* w_int, int n, double scale, int direction,
                                  int n_blocks, void* scratch, double* out, cudaStream_t st)
{
    int C = n / n_blocks / kEstThreads;
    if (C > kEstMaxCtas / n_blocks) C = kEstMaxCtas / n_blocks;
    if (C < 1) C = 1;
    estimator_grid_kernel<<<n_blocks * C, kEstThreads, 0, st>>>(
        w_int, n, scale, direction, n_blocks, C, (double2*)((char*)scratch + 64),
        (unsigned int*)scratch, out);
    return cudaGetLastError();
}

}  // namespace jz
