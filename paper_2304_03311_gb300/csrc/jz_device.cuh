// jz_device.cuh -- device-side building blocks of the replica-gluing kernels.
//
// Spin storage in shared memory (one trajectory per team of threads):
//   S[c][R][q]  uint32 words, c = colour, R = (r L_t + t) L_y + y the row,
//               q < GW = ceil((L/2)/8) the word within the row.  Nibble j of
//               word q holds the colour-c site h = 8q + j of row R, x = 2h + p
//               with p = (c + t + y) mod 2; 0 for spin +1 and 1 for -1.
// With this layout the four (2D) or six (3D) neighbours of the eight sites of
// one word are, in the other colour: the same word of rows t-1, t+1 (and
// y-1, y+1), the same word of the same row (one x neighbour), and that word
// shifted by one nibble (the other x neighbour).  Two Philox4x32-10 blocks
// give the eight acceptance words of one spin word.
#pragma once
#include <cstddef>
#include <cstdint>

namespace jz {

constexpr int kMaxJobsPerLaunch = 4096;
constexpr int kPairTable = 256;   // entries of the acceptance table of site pairs
constexpr size_t kMaxDynSmem = 227 * 1024;   // shared memory of one CTA
// Kept free beside the lattices for that table and the kernels' static arrays.
constexpr size_t kPairReserve = kPairTable * 8 + 512;

// Bounds-checked builds (compiled with -DJZ_BOUNDS_CHECK: the debug library).
// Every lattice access of the trajectory kernels and every label / spin-bit
// access of the Swendsen-Wang kernel checks its index against its array; an
// index outside it sets bit `site` of this translation unit's status word
// (entry 0; entry 1 keeps one offending index) and the access is skipped.
// Release builds compile each check to nothing.
#ifdef JZ_BOUNDS_CHECK
static __device__ unsigned int jz_bounds_status[2];
__device__ __forceinline__ bool in_bounds(long long i, long long n, int site)
{
    if (i >= 0 && i < n) return true;
    atomicOr(&jz_bounds_status[0], 1u << site);
    jz_bounds_status[1] = (unsigned int)i;
    return false;
}
#else
__device__ __forceinline__ bool in_bounds(long long, long long, int) { return true; }
#endif

// Philox4x32-10 round constants and Weyl key increments (Salmon, Moraes, Dror
// and Shaw, SC'11).
constexpr uint32_t kPhiloxM0 = 0xD2511F53u;
constexpr uint32_t kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u;
constexpr uint32_t kPhiloxW1 = 0xBB67AE85u;

// Key schedule of one launch: k0[i], k1[i] for rounds i = 0..9.  Passed by
// value as a kernel parameter, so every round key is a constant-bank operand.
struct PhiloxKeys {
    uint32_t k0[10];
    uint32_t k1[10];
};

// Lattice shape of one launch (all jobs of a launch share it).
struct Geom {
    int L, Lt, Ly;      // spatial extent, time extent, L in 3D / 1 in 2D
    int Lh;             // L / 2 sites of one colour per row
    int G;              // Philox blocks per row, ceil(Lh / 4) (the random-stream layout)
    int GW;             // shared-memory words per row, ceil(Lh / 8) (8 sites per word)
    int nrep;           // replicas n
    int NR;             // rows per colour, n * Lt * Ly
};

// How one launch maps trajectories onto threads: a team of team_threads runs
// one trajectory; a CTA of cta_threads holds `teams` teams.  warp: every team
// lies inside one warp and synchronises with __syncwarp (no cross-warp
// barrier); otherwise the CTA is one team and uses __syncthreads.
struct LaunchShape {
    int team_threads;
    int teams;
    int cta_threads;
    int warp;
};

// How a team's slots (threads per word column) share the n L_t rows: TS slices
// at a time in RS replicas at a time, and the half-sweep's length that follows,
// in twelfths of a bulk row's time.
struct RowSplit {
    int ts, rs, cost;
};

// word: a bulk row's twelfths, 12 for a whole word, 7 for a half one.  A
// thread's first row in each replica costs 8 more (the glued link and the cut
// columns), so splitting the replicas (RS > 1) saves edge rows; it needs TS
// >= 3, where one edge row per replica suffices.  With a whole time column per
// slot (TS = L_t) the rest of the slots are replicas.
__host__ __device__ inline RowSplit split_rows(int slots, int nrep, int Lt, int word)
{
    if (slots >= Lt) {
        const int rs = slots / Lt;
        return RowSplit{Lt, rs, ((nrep + rs - 1) / rs) * (word + 8)};
    }
    RowSplit b{slots, 1, nrep * (word * ((Lt + slots - 1) / slots) + (slots == 1 ? 16 : 8))};
    for (int rs = 2; rs <= nrep && slots / rs >= 3; ++rs) {
        const int ts = slots / rs;
        const int cost = ((nrep + rs - 1) / rs) * (word * ((Lt + ts - 1) / ts) + 8);
        if (cost < b.cost) b = RowSplit{ts, rs, cost};
    }
    return b;
}

// How a team works on a row's words: all alike, whole ones (kWhole) or the last
// one ragged (kRagged); or, when the last word has at most four sites and needs
// one Philox block only, these half words apart from the others (kHalfTail).
enum RowKind { kRagged = 0, kWhole = 1, kHalfTail = 2 };

// A half-sweep's length with a team of nthr threads (split_rows' unit), and the
// kind it takes: half words apart where that is shorter.  In short half-sweeps, up to
// six rows per thread (kShortSweep), a second pass over the half-sweep counts as well
// (kSecondPass, an edge row's extra): up to 152 trajectories of 3D L = 18 .. 24, L_t = 2
// .. 24, at 35 against 40 or 73 against 80 units, take 0.78 .. 0.95 of the time in one pass
// (L = 22, 24, L_t = 6: 1.02); 300 of L = 18, L_t = 4, where throughput counts, 1.04.  3D L =
// 36, 40, L_t = 16, at 109 against 112 units, take 1.05 in one pass.
constexpr int kSecondPass = 8, kShortSweep = 80;
__host__ __device__ inline int sweep_cost(const Geom& g, int nthr, RowKind* kind)
{
    const int all = split_rows(nthr / (g.GW * g.Ly), g.nrep, g.Lt, 12).cost;
    *kind = g.Lh % 8 == 0 ? kWhole : kRagged;
    if (g.Lh % 8 == 0 || g.Lh % 8 > 4) return all;
    const int whole =
        g.GW == 1 ? 0 : split_rows(nthr / ((g.GW - 1) * g.Ly), g.nrep, g.Lt, 12).cost;
    const int apart = whole + split_rows(nthr / g.Ly, g.nrep, g.Lt, 7).cost;
    if (apart + (whole && all <= kShortSweep ? kSecondPass : 0) < all) *kind = kHalfTail;
    return all < apart ? all : apart;
}
__host__ __device__ inline RowKind row_kind(const Geom& g, const LaunchShape& sh)
{
    RowKind k;
    sweep_cost(g, sh.team_threads, &k);
    return k;
}

// A team with a thread per spin word of its lattice.  Where it is a warp team and L =
// 16 in 2D (kernels of compile-time GW = 1), it runs the one-row path (run_rows).
__host__ __device__ inline bool one_row_team(const Geom& g, const LaunchShape& sh)
{
    return sh.team_threads == g.NR * g.GW;
}

// Per-job (one transformation) parameters, device copy.
struct JobDesc {
    int l;              // switched column
    int n_step, n_sweep, n_therm;
    int dir;            // +1 forward, -1 reverse
    int n_traj;
    int prot;           // 1: every switched column together; 2: one column y at a time
    int g0, g1;         // columns x < g0 glued, g0 <= x < g1 switching, x >= g1 self
    int k_begin, k_end; // protocol steps run: [k_begin, k_end); 0 starts from the hot start
    int start_in;       // 1: step k_begin = 0 starts from spins_in (thermalised elsewhere)
    const int8_t* spins_in;     // k_begin > 0 or start_in: [n_traj][V] state after step k_begin - 1
    const long long* w_in;      // k_begin > 0: [n_traj] W_int of steps 0 .. k_begin - 1
    long long traj0;    // global index of the job's first trajectory
    long long cta0;     // first CTA of the job in the launch grid
    uint32_t tb[4];     // bulk thresholds by anti-aligned neighbour count a:
                        // tb[a] = T(m = 2D - 2a), a < D
    int weak;           // 1: a threshold of tcut with m > 0 may round up to 2^32 - 1
    const uint32_t* tcut;   // [n_step][8D] switched-site thresholds
    long long* w_out;       // [n_traj] W_int
    int8_t* spins_out;      // [n_traj][V] final spins (+-1) or nullptr
};

// One job of a persistent batch launch.
struct BatchJob {
    JobDesc J;            // thresholds, outputs, trajectory range
    Geom g;
    int D, kind;          // RowKind
    LaunchShape sh;       // team size, teams per CTA (= trajectories per work item), barrier
    int lattice_words;    // 2 * NR * GW spin words per team
};

// One job of the batched estimator.
struct EstJob {
    const long long* w;   // n work values W_int
    int n;
    int direction;
    int n_blocks;         // jackknife blocks, <= 64 and <= n
    double scale;         // beta / N
};

// One Philox4x32-10 block.
__device__ __forceinline__ uint4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                        const PhiloxKeys& K)
{
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        const uint64_t p0 = (uint64_t)kPhiloxM0 * c0;
        const uint64_t p1 = (uint64_t)kPhiloxM1 * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ K.k0[i];
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ K.k1[i];
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
        c0 = n0;
        c2 = n2;
    }
    return make_uint4(c0, c1, c2, c3);
}

// The block whose counter entering round R is (c0, c1, c2, c3).
template <int R>
__device__ __forceinline__ uint4 philox_from(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                             const PhiloxKeys& K)
{
#pragma unroll
    for (int i = R; i < 10; ++i) {
        const uint64_t q0 = (uint64_t)kPhiloxM0 * c0;
        const uint64_t q1 = (uint64_t)kPhiloxM1 * c2;
        const uint32_t n0 = (uint32_t)(q1 >> 32) ^ c1 ^ K.k0[i];
        const uint32_t n2 = (uint32_t)(q0 >> 32) ^ c3 ^ K.k1[i];
        c1 = (uint32_t)q1;
        c3 = (uint32_t)q0;
        c0 = n0;
        c2 = n2;
    }
    return make_uint4(c0, c1, c2, c3);
}

// One block with round 0's product (hi1, lo1) = M1 * c2 supplied: counter word
// 2 is the trajectory index, fixed for a whole trajectory.
__device__ __forceinline__ uint4 philox_r0(uint32_t c0, uint32_t c1, uint32_t hi1, uint32_t lo1,
                                           uint32_t c3, const PhiloxKeys& K)
{
    const uint64_t p0 = (uint64_t)kPhiloxM0 * c0;
    return philox_from<1>(hi1 ^ c1 ^ K.k0[0], lo1, (uint32_t)(p0 >> 32) ^ c3 ^ K.k1[0],
                          (uint32_t)p0, K);
}

// Sum of v over a warp, in every lane.
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// The last stage of the FP64 estimator of one job (Appendix A, eq.
// Jarzynski_theorem; blocked jackknife), given each jackknife block's maximum
// m_b of -W_i and shifted sum s_b = sum_i e^{-W_i - m_b} (rows lo[b] ..
// lo[b+1] - 1, B <= 64 blocks): the estimate without each block b and the full
// one as max-shifted log-sum-exps over the blocks; thread 0 writes out[0] = ln
// <e^-W>, out[1] = Delta S, out[2] = the jackknife error.  Every thread of the
// CTA, at least kEstFinish of them, calls it (it holds barriers); s_exp: 2 B words
// of shared memory.
//
// What bounds it: one CTA's chain of FP64 operations at GB300's FP64 rate (two
// lanes per clock and SM).  The maximum without block b is the overall one
// unless block b alone holds it, so only two sets of B exponentials exist; one
// thread forms each, four (B <= 32) or two threads share an estimate's sum, its
// two logarithms run in two lanes, and the maxima compare as integers.
constexpr int kEstFinish = 160;
__device__ __forceinline__ void estimator_finish(const double* s_max, const double* s_sum,
                                                 const int* s_lo, int B, int n, int direction,
                                                 double* s_theta, double* s_exp, double* out)
{
    const int t = (int)threadIdx.x, lane = t & 31;
    // every warp: the largest block maximum, its block, the largest of the rest
    auto key = [](double v) {   // order-preserving
        const long long k = __double_as_longlong(v);
        return k ^ ((k >> 63) & 0x7FFFFFFFFFFFFFFFLL);
    };
    const long long none = key(-INFINITY);
    long long k1 = lane < B ? key(s_max[lane]) : none;
    long long k2 = lane + 32 < B ? key(s_max[lane + 32]) : none;
    int top = lane;
    if (k2 > k1) {
        const long long x = k1;
        k1 = k2;
        k2 = x;
        top = lane + 32;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long a1 = __shfl_xor_sync(0xFFFFFFFFu, k1, o);
        const long long a2 = __shfl_xor_sync(0xFFFFFFFFu, k2, o);
        const int at = __shfl_xor_sync(0xFFFFFFFFu, top, o);
        const bool up = a1 > k1 || (a1 == k1 && at < top);
        const long long lower = up ? k1 : a1;
        k2 = lower > k2 ? lower : k2;
        k2 = a2 > k2 ? a2 : k2;
        k1 = up ? a1 : k1;
        top = up ? at : top;
    }
    auto val = [](long long k) {
        return __longlong_as_double(k ^ ((k >> 63) & 0x7FFFFFFFFFFFFFFFLL));
    };
    const double m1 = val(k1), m2 = val(k2);
    if (t < B) s_exp[t] = exp(s_max[t] - m1);
    if (t >= 64 && t - 64 < B) s_exp[B + t - 64] = t - 64 == top ? 0.0 : exp(s_max[t - 64] - m2);
    __syncthreads();
    const int P = B <= 32 ? 4 : 2;
    const int est = t / P, part = t - est * P;
    double tot = 0.0;
    if (est <= B) {
        const double* e = est == top ? s_exp + B : s_exp;
        for (int b = part; b < B; b += P)
            if (b != est) tot += s_sum[b] * e[b];
    }
    for (int o = P / 2; o > 0; o >>= 1) tot += __shfl_xor_sync(0xFFFFFFFFu, tot, o);
    // lane `part` 0 takes ln of the sum, 1 that of the row count
    const int count = est < B ? n - (s_lo[est + 1] - s_lo[est]) : n;
    const double ln = est <= B && part < 2 ? log(part ? (double)count : tot) : 0.0;
    const double ln_count = __shfl_xor_sync(0xFFFFFFFFu, ln, 1);
    if (est <= B && part == 0) s_theta[est] = (est == top ? m2 : m1) + ln - ln_count;
    __syncthreads();
    if (t >= 32) return;
    const double sign = direction > 0 ? -1.0 : 1.0;
    const double full = s_theta[B];
    double err = 0.0;
    if (B >= 2) {
        const double a = lane < B ? sign * s_theta[lane] : 0.0;
        const double b = lane + 32 < B ? sign * s_theta[lane + 32] : 0.0;
        const double mean = warp_sum(a + b) / B;
        const double da = lane < B ? a - mean : 0.0, db = lane + 32 < B ? b - mean : 0.0;
        err = sqrt((double)(B - 1) / B * warp_sum(da * da + db * db));
    }
    if (t != 0) return;
    out[0] = full;
    out[1] = sign * full;
    out[2] = err;
}

__device__ __forceinline__ uint32_t word_of(const uint4& u, int j)
{
    return j == 0 ? u.x : j == 1 ? u.y : j == 2 ? u.z : u.w;
}

}  // namespace jz
