// jz_traj_kernel.cuh -- the per-trajectory kernel of the Jarzynski
// replica-gluing method (jz_traj.cuh) and its instantiations' selectors; one
// translation unit per dimension compiles them.
#pragma once
#include <cstdint>

#include "jz_device.cuh"
#include "jz_traj.cuh"

namespace jz {

// Finds the job owning CTA b: the last j with jobs[j].cta0 <= b.
__device__ __forceinline__ int find_job(const JobDesc* __restrict__ jobs, int n_jobs, long long b)
{
    int lo = 0, hi = n_jobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&jobs[mid].cta0) <= b) lo = mid; else hi = mid - 1;
    }
    return lo;
}

constexpr int kMaxTeams = 64;

// One CTA runs `teams` trajectories of the job that owns it (sh.teams per
// CTA; warp teams sync with __syncwarp, a CTA team with __syncthreads).  The
// lattices live in shared memory, behind PAIR's acceptance table, or, when they
// do not fit there (HBM), in this CTA's own slice of an HBM buffer (L1/L2-cached).
//
// Registers: up to 128, i.e. 16 warps per SM.  The update is bound by the
// arithmetic pipes, not by latency: capped at 96, 80, 72 and 64 registers (20
// to 32 warps) the 2D L = 64 scan (31 x 1024 trajectories) took 0.99, 1.00, 1.05
// and 1.06 of the time uncapped, the 3D L = 24, L_t = 96 lattice 0.99, 1.06, 1.16
// and 1.16.
template <int D, int KIND, bool PAIR, int CW, int CLY, bool WARP, bool HBM, int CLT = 0,
          int CTS = 0>
__global__ void __launch_bounds__(512, 1)
traj_kernel(const Geom g, const PhiloxKeys K, const JobDesc* __restrict__ jobs, int n_jobs,
            const LaunchShape sh, uint32_t* __restrict__ gS)
{
    extern __shared__ uint2 s_dyn[];
    uint2* s_tab = s_dyn;
    uint32_t* S = HBM ? gS + (size_t)blockIdx.x * sh.teams * (2 * g.NR * g.GW)
                      : (uint32_t*)(s_dyn + (PAIR ? kPairTable : 0));
    __shared__ int s_work[kMaxTeams];

    const int j = find_job(jobs, n_jobs, (long long)blockIdx.x);
    const JobDesc& J = jobs[j];
    const TeamJob tj = team_job(J, g.Ly);
    const long long cta_local = (long long)blockIdx.x - __ldg(&J.cta0);
    int team, tid;
    team_of(sh, &team, &tid);
    const long long local = cta_local * sh.teams + (team < 0 ? 0 : team);
    const bool has = team >= 0 && local < __ldg(&J.n_traj);
    if (!has) tid = -1;
    const int tm = team < 0 ? 0 : team;
    uint32_t* St = S + (size_t)tm * (2 * g.NR * g.GW);
    if (PAIR) fill_pairs<D>(s_tab, J.tb);
    for (int i = threadIdx.x; i < kMaxTeams; i += blockDim.x) s_work[i] = 0;
    __syncthreads();
    const long long traj = __ldg(&J.traj0) + local;
    const long long V = (long long)g.nrep * g.Lt * g.Ly * g.L;
    const int8_t* sin = (has && (tj.k_begin > 0 || tj.start_in)) ? J.spins_in + local * V : nullptr;
    int dE;
    // The one-row path is compiled into the 2D GW = 1 variant (L = 16), the
    // only lattice whose warp team can hold a thread per word.
    constexpr bool kRow = D == 2 && KIND == kWhole && CW == 1 && WARP;
    if (kRow && one_row_team(g, sh))
        dE = run_trajectory<D, KIND, PAIR, HBM, CW, CLY, kRow>(g, K, tj, traj, St, s_tab, tid,
                                                               sh.team_threads, WarpBarrier{}, sin);
    else if (WARP)
        dE = run_trajectory<D, KIND, PAIR, HBM, CW, CLY, false, CLT, CTS>(
            g, K, tj, traj, St, s_tab, tid, sh.team_threads, WarpBarrier{}, sin);
    else
        dE = run_trajectory<D, KIND, PAIR, HBM, CW, CLY>(g, K, tj, traj, St, s_tab, tid,
                                                         sh.team_threads, CtaBarrier{}, sin);
    if (has && dE != 0) atomicAdd(&s_work[tm], dE);
    __syncthreads();
    if (has && tid == 0)
        J.w_out[local] = (tj.k_begin > 0 ? J.w_in[local] : 0) +
                         (long long)(tj.dir > 0 ? s_work[tm] : -s_work[tm]) *
                             (tj.prot == 2 ? g.Ly : 1);
    int8_t* sp = J.spins_out;
    if (has && sp != nullptr) export_spins<D>(g, St, sp + local * V, tid, sh.team_threads);
}

using TrajFn = void (*)(const Geom, const PhiloxKeys, const JobDesc*, int, const LaunchShape,
                       uint32_t*);

template <int D, int KIND, bool PAIR, int CW, int CLY, int CLT = 0, int CTS = 0>
TrajFn pick_traj(const LaunchShape& sh, bool hbm)
{
    return hbm ? (sh.warp ? traj_kernel<D, KIND, PAIR, CW, CLY, true, true>
                          : traj_kernel<D, KIND, PAIR, CW, CLY, false, true>)
               : (sh.warp ? traj_kernel<D, KIND, PAIR, CW, CLY, true, false, CLT, CTS>
                          : traj_kernel<D, KIND, PAIR, CW, CLY, false, false>);
}

// The instantiation that runs lattices g in shape sh (pair: with the
// acceptance table, see traj_pairs): jz_traj2d.cu, jz_traj3d.cu.
TrajFn select_traj2d(const Geom& g, const LaunchShape& sh, bool hbm, bool pair);
TrajFn select_traj3d(const Geom& g, const LaunchShape& sh, bool hbm, bool pair);

}  // namespace jz
