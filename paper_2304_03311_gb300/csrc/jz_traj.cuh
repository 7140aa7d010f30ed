// jz_traj.cuh -- one Jarzynski trajectory of the replica-gluing method, run
// by a team of threads over a replica lattice held in shared memory.
//
// Per trajectory (section 3, linear protocol; Appendix A, eq.
// work_in_one_MC_step and the remark on the update at lambda_{k+1}): hot
// start, n_therm checkerboard Metropolis sweeps at the start geometry, then N
// protocol steps, each the work increment dE_k on phi_k followed by n_sweep
// sweeps at lambda_{k+1}.
//
// Layout: S[colour][row R][word q], R = (r L_t + t) L_y + y, q < GW = ceil(L/16);
// nibble j (bits 4j..4j+3) of word q is the colour-c site h = 8q + j of the
// row, x = 2h + p, p = (c + t + y) mod 2, value 0 for spin +1 and 1 for -1.
// A word's eight sites draw from Philox blocks 2q and 2q+1 of their row.
// Nibble-wise sums of the neighbours' words give the number of neighbours of
// spin -1 of all eight sites at once (at most 6, so no carries cross nibbles).
//
// Team mapping: the team's threads per word column are TS x RS slots; thread
// (r0, t0, y, q) owns word q of row y of every TS-th time slice in the replicas
// r0, r0 + RS, ... and both colours, so all its index and wrap arithmetic is
// fixed.  split_rows chooses TS and RS for the shortest half-sweep.  A replica's
// rows are one or two edge rows per thread, which blend in the glued replica and
// handle the switched columns (half_sweep says which rows), and bulk rows; an
// edge row costs about 90 instructions more, so two replicas on two sets of
// slots, one edge row per thread, beat one set that has two (2D L = 128, L_t =
// 1024 CTA teams: 109.7 -> 106.8 ms per 8-column scan).  Where the last word of
// a row holds at most four sites, i.e. draws one Philox block, and it pays
// (sweep_cost), these half words are shared out apart from the whole ones, and
// no thread draws a block that no site uses (3D L = 24, L_t = 96: 121.4 -> 103.0
// ms).  CW, CLY > 0 fix GW and L_y at compile time (neighbour loads then use
// immediate offsets); 0 reads them from Geom.
//
// What bounds it (ncu and instruction-mix probes on GB300, cycles per SM
// sub-partition and spin word of 32 lanes): the pipes that issue the two
// Philox blocks of a word and its update.  A 32 x 32 -> 64-bit multiply holds
// the FMA pipe for 4 cycles and a result port that it shares with the 2-cycle
// logic and add instructions for 2; the bare Philox of a word (34 multiplies, 38
// three-input XORs) takes 143 cycles, every further ALU instruction adds about
// 1.8, every multiply-add 1.4, every shared load about 1.  So the update is
// written for few instructions of any kind: thresholds looked up for two sites
// at once, sums instead of XORs, one funnel shift per word, wrap-free bulk rows.
// 2D L = 64: 130 instructions and 216 cycles per word (158 and 314 with one lookup per
// site, four copies of the half-sweep whose code overflowed the instruction cache, and a
// cut pass that recomputed its geometry): a scan of 31 x 1024 trajectories 761 -> 523 ms,
// 1.02e12 -> 1.49e12 spin updates/s, at 2.07 GHz.
//
// The work increment is gathered inside the first colour-0 half-sweep of each
// step: for every (r, y) exactly one of the switched sites (l, y, 0)^r and
// (l, y, 1)^r has colour 0, and s_i (s_self - s_glue) summed over those sites
// equals sum_{r,y} s^r(l,y,0) [s^r(l,y,1) - s^{r+1}(l,y,1)] (re-index the glue
// sum over r).  Each such site's own thread reads these values before it
// updates, and only colour-1 sites enter the products, so no extra barrier is
// needed.
#pragma once
#include <cstdint>

#include "jz_device.cuh"

namespace jz {

// ------------------------------------------------------------- acceptance --
// A site with a anti-aligned neighbours (energy cost m = 2D - 2a) flips when
// a >= D, else iff its draw is below tb[a] = T(m).

// f += 2^SH if u <= t: one compare and one predicated add.
template <int SH>
__device__ __forceinline__ void add_if_le(uint32_t& f, uint32_t u, uint32_t t)
{
    asm("{.reg .pred q; setp.le.u32 q, %1, %2; @q add.u32 %0, %0, %3;}"
        : "+r"(f)
        : "r"(u), "r"(t), "n"((int)(1u << SH)));
}
// f += 2^SH if u < t.
template <int SH>
__device__ __forceinline__ void add_if_lt(uint32_t& f, uint32_t u, uint32_t t)
{
    asm("{.reg .pred q; setp.lt.u32 q, %1, %2; @q add.u32 %0, %0, %3;}"
        : "+r"(f)
        : "r"(u), "r"(t), "n"((int)(1u << SH)));
}

// PAIR acceptance, the form of every job that allows it: a 256-entry table of
// threshold pairs in shared memory, indexed by one byte of v, i.e. by two sites at once.  Nibble j of v is site
// j's state: its neighbours of spin -1 counted (at most 2D < 8), its own spin in
// bit 3.  A site flips iff its draw is at most its threshold.  Returns the flip
// bits (bit 4j); sites 0..3 use the words of block ua, sites 4..7 those of ub (HALF:
// a word of at most four sites).
template <bool HALF>
__device__ __forceinline__ uint32_t accept_pairs(uint32_t v, const uint4& ua, const uint4& ub,
                                                 const uint2* tab)
{
    const uint2 t01 = tab[v & 0xFFu];
    const uint2 t23 = tab[__byte_perm(v, 0, 0x4441)];
    uint32_t f = 0;
    add_if_le<0>(f, ua.x, t01.x);
    add_if_le<4>(f, ua.y, t01.y);
    add_if_le<8>(f, ua.z, t23.x);
    add_if_le<12>(f, ua.w, t23.y);
    if (HALF) return f;
    const uint2 t45 = tab[__byte_perm(v, 0, 0x4442)];
    const uint2 t67 = tab[v >> 24];
    add_if_le<16>(f, ub.x, t45.x);
    add_if_le<20>(f, ub.y, t45.y);
    add_if_le<24>(f, ub.z, t67.x);
    add_if_le<28>(f, ub.w, t67.y);
    return f;
}

// The table of one job, filled by the CTA's threads: "at most tb[a] - 1", or
// "always" (a >= D).  It cannot say "never" (tb[a] = 0, strong couplings): such
// jobs take the counts below.
template <int D>
__device__ __forceinline__ void fill_pairs(uint2* tab, const uint32_t* __restrict__ tb)
{
    auto at = [&](int v) {
        const int s = v & 7;
        const int a = (v & 8) ? 2 * D - s : s;
        if (a < 0 || a >= D) return 0xFFFFFFFFu;
        return __ldg(tb + a) - 1u;
    };
    for (int i = threadIdx.x; i < kPairTable; i += blockDim.x)
        tab[i] = make_uint2(at(i & 15), at(i >> 4));
}

// COUNT acceptance, for jobs without a table (a threshold of zero, or no shared
// memory left beside the lattice) and for run_rows, where the counts are off the
// path from one half-sweep to the next: 2D, 4 instructions per site against the
// table's 3.5 (3D: 6).  Nibble j of the result is the number of thresholds T[i],
// i < D, above site j's draw.  tb grows with a, so the site flips iff
// a + count >= D.  It depends on the draws alone.
template <int D, bool HALF = false>
__device__ __forceinline__ uint32_t count8(const uint4& ua, const uint4& ub, const uint32_t* T)
{
    uint32_t n = 0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        add_if_lt<0>(n, ua.x, T[i]);
        add_if_lt<4>(n, ua.y, T[i]);
        add_if_lt<8>(n, ua.z, T[i]);
        add_if_lt<12>(n, ua.w, T[i]);
        if (HALF) continue;
        add_if_lt<16>(n, ub.x, T[i]);
        add_if_lt<20>(n, ub.y, T[i]);
        add_if_lt<24>(n, ub.z, T[i]);
        add_if_lt<28>(n, ub.w, T[i]);
    }
    return n;
}

// The flip bits from the counts n, the nibble-wise sums s of the neighbours of
// spin -1 and the own spins: with a = s (own 0) or 2D - s (own 1), the new
// spin is [s + n >= D] or [s - n >= D + 1], and 3 - n = n ^ 3, so both are
// bit 3 of one nibble-wise sum (between 1 and 14: no carries).
template <int D>
__device__ __forceinline__ uint32_t flips_of_counts(uint32_t s, uint32_t own, uint32_t n)
{
    const uint32_t x = s + (n ^ (own * 3u)) - own * 4u + (uint32_t)(8 - D) * 0x11111111u;
    return ((x >> 3) & 0x11111111u) ^ own;
}

__device__ __forceinline__ uint32_t word8(const uint4& ua, const uint4& ub, int j)
{
    return word_of(j < 4 ? ua : ub, j & 3);
}

// The words of a row that a thread set owns: all of them, or, where rows end in
// half a word, the whole words and the half words apart.
enum RowPart { kAllWords = 0, kWholeWords = 1, kTailWords = 2 };

// Per-job values a team needs (read from the job descriptor once).
struct TeamJob {
    int l, n_step, n_sweep, n_therm, dir;
    int k_begin, k_end;   // protocol steps run; k_begin > 0 resumes from stored spins
    int start_in;         // 1: step k_begin = 0 starts from stored (thermalised) spins
    int g0, g1;   // columns x < g0 glued, g0 <= x < g1 switching, x >= g1 self
    int prot;     // 1: every switched column together; 2: one column y at a time
    int den;      // steps of one column's run: N (protocol 1), N / L_y (protocol 2)
    const uint32_t* tcut;
    uint32_t tb[3];       // bulk thresholds, a < D
    bool weak;            // a switched threshold of m > 0 may round up to 2^32 - 1
};

// What a row's update needs beside its words: the protocol step (k < 0: none)
// and its weights.
struct StepState {
    int k, lg, w_self, w_glue;
    const uint32_t* tk;   // step k's switched-site thresholds
    bool record;
};

// Where a team's lattice lies: byte addresses of its words, 32-bit ones in
// shared memory (one add per address, immediate offsets folded into the
// access) or pointers into an HBM slice.
template <bool HBM>
struct Mem;
template <>
struct Mem<false> {
    using A = uint32_t;
    static __device__ __forceinline__ A at(uint32_t* p)
    {
        return (uint32_t)__cvta_generic_to_shared(p);
    }
    static __device__ __forceinline__ uint32_t ld(A a)
    {
        uint32_t v;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
        return v;
    }
    static __device__ __forceinline__ void st(A a, uint32_t v)
    {
        asm volatile("st.shared.u32 [%0], %1;" : : "r"(a), "r"(v) : "memory");
    }
};
template <>
struct Mem<true> {
    using A = char*;
    static __device__ __forceinline__ A at(uint32_t* p) { return (char*)p; }
    static __device__ __forceinline__ uint32_t ld(A a) { return *(const uint32_t*)a; }
    static __device__ __forceinline__ void st(A a, uint32_t v) { *(uint32_t*)a = v; }
};

// CLT, CTS > 0: L_t and the slice step TS fixed at compile time (the 2D L = 64,
// L_t = 64 warp teams); 0 reads them from Geom and the team size.
template <int D, bool FAST, bool PAIR, bool HBM, int CW = 0, int CLY = 0, int CLT = 0, int CTS = 0,
          int PART = kAllWords>
struct Traj {
    static constexpr bool HALF = PART == kTailWords;
    using M = Mem<HBM>;
    using A = typename M::A;
    // A thread's edge row (t = 0, 1 next to the cut, or any other, whose
    // neighbour "across" is its t + 1 row): byte offsets that hold for a whole
    // trajectory.
    struct Edge {
        int t;            // the row
        int n, x;         // the ordinary time neighbour; the row across
        int g, gw, rw;    // the glued partner across: + g, in replica rw + gw
    };

    const Geom& g;
    uint32_t* S;              // this team's spin words [2][NR * GW]
    A S0;                     // their address
    const uint2* tab;         // PAIR: the job's threshold pairs
    const TeamJob& J;
    const PhiloxKeys& K;
    uint32_t hi1, lo1;        // M1 * traj: round 0 of Philox for counter word 2
    uint32_t c3base;          // dir bit << 1 | l << 2
    int q, y, t0, TS;         // this thread's word, row y, first slice and slice step
    int r0, RS;               // first replica and replica step
    int d_qm, d_qp;           // byte offset of the x-shift neighbour word (p = 0 / 1)
    int d_ym, d_yp;           // byte offsets of the rows y-1 / y+1 (3D)
    Edge edge;                // TS >= 2: the first row of each replica
    int tb, n_all, up_last;   // first bulk row, the rows all slots have, the last one's t + 1 row
    bool has_last;            // one row more
    uint32_t vmask;           // nibbles of word q that hold sites (ragged rows)
    int sh_next, sh_prev;     // ragged rows: nibble position of the wrapped x neighbour

    __device__ __forceinline__ int W() const { return CW > 0 ? CW : g.GW; }
    __device__ __forceinline__ int Ly() const { return D == 2 ? 1 : (CLY > 0 ? CLY : g.Ly); }
    __device__ __forceinline__ int rowW() const { return Ly() * W(); }
    // words of a row that this thread set owns, from word first() on
    __device__ __forceinline__ int own_words() const
    {
        return PART == kAllWords ? W() : PART == kWholeWords ? W() - 1 : 1;
    }
    __device__ __forceinline__ int first() const { return HALF ? W() - 1 : 0; }
    __device__ __forceinline__ int Lt() const { return CLT > 0 ? CLT : g.Lt; }
    // Philox blocks per row: full words have two each
    __device__ __forceinline__ int G() const { return CW > 0 && FAST ? 2 * CW : g.G; }
    __device__ __forceinline__ int step() const { return CTS > 0 ? CTS : TS; }

    // The word at address a, of the colour starting at base (checked in
    // bounds-checked builds: a word outside the colour is recorded and the
    // access skipped).
    __device__ __forceinline__ uint32_t ld(A base, A a, int site) const
    {
        return in_bounds((long long)(a - base) >> 2, (long long)g.NR * g.GW, site) ? M::ld(a) : 0u;
    }
    __device__ __forceinline__ void st(A base, A a, uint32_t v, int site) const
    {
        if (in_bounds((long long)(a - base) >> 2, (long long)g.NR * g.GW, site)) M::st(a, v);
    }
    __device__ __forceinline__ A colour(int c) const { return S0 + c * (g.nrep * Lt() * rowW() * 4); }

    // tid < 0: a thread with no sites (it still takes part in the barriers).
    __device__ __forceinline__ Traj(const Geom& g_, uint32_t* S_, const uint2* tab_,
                                    const TeamJob& J_, const PhiloxKeys& K_, uint32_t traj,
                                    int tid, int nthr)
        : g(g_), S(S_), S0(M::at(S_)), tab(tab_), J(J_), K(K_)
    {
        c3base = ((uint32_t)(J.dir < 0) << 1) | ((uint32_t)J.l << 2);
        const uint64_t p1 = (uint64_t)kPhiloxM1 * traj;
        hi1 = (uint32_t)(p1 >> 32);
        lo1 = (uint32_t)p1;
        const int wp = own_words();
        if (wp == 0) tid = -1;   // rows of half a word have no whole one
        const int col = max(wp, 1) * Ly();
        const int slots = nthr / col;   // threads per word column
        const RowSplit sp = split_rows(slots, g.nrep, g.Lt, HALF ? 7 : 12);
        TS = CTS > 0 ? CTS : sp.ts;
        RS = CTS > 0 ? slots / CTS : sp.rs;
        if (tid < 0 || tid / col >= TS * RS) {
            q = y = 0;
            t0 = g.Lt;
            r0 = g.nrep;
        } else {
            q = first() + tid % wp;
            y = (tid / wp) % Ly();
            t0 = (tid / col) % TS;
            r0 = (tid / col) / TS;
        }
        d_qm = 4 * ((q == 0 ? W() - 1 : q - 1) - q);
        d_qp = 4 * ((q == W() - 1 ? 0 : q + 1) - q);
        d_ym = 4 * ((y == 0 ? Ly() - 1 : y - 1) - y) * W();
        d_yp = 4 * ((y == Ly() - 1 ? 0 : y + 1) - y) * W();
        const int nv = g.Lh - 8 * q;                       // sites in this word
        const int nv_last = g.Lh - 8 * (W() - 1);          // sites in the row's last word
        vmask = nv >= 8 ? 0xFFFFFFFFu : ((1u << (4 * nv)) - 1u);
        sh_next = 4 * ((nv >= 8 ? 8 : nv) - 1);
        sh_prev = q == 0 ? 4 * (nv_last - 1) : 28;
        const bool rot = step() >= 3;
        edge = edge_of(!rot ? t0 : t0 == 0 ? Lt() - 1 : t0 - 1);
        tb = rot ? t0 - 1 + step() : (step() == 1 ? 2 : t0 + 2);
        const int end = rot ? Lt() - 1 : Lt();
        const int n = tb < end ? (end - tb - 1) / step() + 1 : 0;
        // every slot has n_all or (L_t and L even) n_all + 1 bulk rows
        n_all = (rot ? (Lt() + step() - 1) / step() - 1 : n) - 1;
        has_last = n > n_all;
        up_last = 4 * rowW() * (!rot && tb + (n - 1) * step() == Lt() - 1 ? -(Lt() - 1) : 1);
    }

    // Flip bits of a word: s = nibble-wise sums of the neighbours of spin -1.
    __device__ __forceinline__ uint32_t flips(uint32_t s, uint32_t own, const uint4& ua,
                                              const uint4& ub) const
    {
        if constexpr (PAIR) {
            return accept_pairs<HALF>(s + own * 8u, ua, ub, tab);
        } else {
            return flips_of_counts<D>(s, own, count8<D, HALF>(ua, ub, J.tb));
        }
    }

    // Glue mask: nibbles of word q (row parity p) whose site has x < lg.
    __device__ __forceinline__ uint32_t glue_mask(int lg, int p) const
    {
        int nj = ((lg - p + 1) >> 1) - 8 * q;   // # of sites 2h + p < lg in this word
        nj = nj < 0 ? 0 : (nj > 8 ? 8 : nj);
        return nj == 8 ? 0xFFFFFFFFu : ((1u << (4 * nj)) - 1u);
    }

    // The x neighbour not at the same h -- h - 1 for p = 0, h + 1 for p = 1 -- of
    // a word's eight sites, out of two words of the other colour's row: lo (at
    // offset a) shifted down by s, joined by hi (at offset b) above it.
    struct XShift {
        int a, b;
        uint32_t s, m;   // FAST: a funnel shift by s; ragged: (lo >> s) + hi m
    };
    __device__ __forceinline__ XShift xshift(int p) const
    {
        XShift x;
        x.a = p ? 0 : d_qm;
        x.b = p ? d_qp : 0;
        if (FAST) {
            x.s = p ? 4u : 28u;
            x.m = 0;
        } else {
            // words hold no bits beyond their sites, so lo >> s leaves one
            // nibble (p = 0) or clears the last one (p = 1)
            x.s = p ? 4u : (uint32_t)sh_prev;
            x.m = p ? 1u << sh_next : 16u;
        }
        return x;
    }
    __device__ __forceinline__ uint32_t xjoin(uint32_t lo, uint32_t hi, const XShift& x) const
    {
        return FAST ? __funnelshift_r(lo, hi, x.s) : (lo >> x.s) + hi * x.m;
    }

    // What the two Philox blocks of every word of a half-sweep share: the rounds
    // 0 and 1 up to the block index (counter word 0).
    struct Stream {
        uint32_t c3k, lo1k, h0k, l0;
    };
    __device__ __forceinline__ Stream stream(int c, uint32_t sweep) const
    {
        const uint64_t q0 = (uint64_t)kPhiloxM0 * (hi1 ^ sweep ^ K.k0[0]);
        Stream x;
        x.c3k = ((uint32_t)c | c3base) ^ K.k1[0];
        x.lo1k = lo1 ^ K.k0[1];
        x.h0k = (uint32_t)(q0 >> 32) ^ K.k1[1];
        x.l0 = (uint32_t)q0;
        return x;
    }
    // The block whose round 0 product is p0 = M0 * (block index).
    __device__ __forceinline__ uint4 draw(uint64_t p0, const Stream& x) const
    {
        const uint64_t q1 = (uint64_t)kPhiloxM1 * ((uint32_t)(p0 >> 32) ^ x.c3k);
        return philox_from<2>((uint32_t)(q1 >> 32) ^ x.lo1k, (uint32_t)q1,
                              x.h0k ^ (uint32_t)p0, x.l0, K);
    }

    // The word's second block; a half word has none.
    __device__ __forceinline__ uint4 second(uint64_t p0, const Stream& x) const
    {
        return HALF ? make_uint4(0u, 0u, 0u, 0u) : draw(p0 + kPhiloxM0, x);
    }

    // Site jl of a cut-row word that switches during the protocol: couplings
    // beta (1 - lambda) to its own replica (self_w), beta lambda to the next
    // one (glue_w), tested against step k's table; returns its flip bit.  s:
    // nibble-wise sums of its neighbours of spin -1, the self link's among them.
    // With z = 4 (fixed links' sum) + 2 self + glue the table's index is z for
    // a spin -1, 8D - 1 - z for a spin +1.  record: add its share of dE_k.
    __device__ __forceinline__ uint32_t switched_site(int jl, uint32_t own, uint32_t self_w,
                                                      uint32_t glue_w, uint32_t s, uint32_t u,
                                                      const StepState& P, int& dE) const
    {
        const int sh = 4 * jl;
        const bool ob = (own >> sh) & 1u;
        const int sf = (int)((self_w >> sh) & 1u), gl = (int)((glue_w >> sh) & 1u);
        const int z = 4 * (int)((s >> sh) & 7u) - 2 * sf + gl;
        const int ti = ob ? z : 8 * D - 1 - z;
        const uint32_t T = __ldg(P.tk + ti);
        // m <= 0 (always) is stored as 2^32 - 1, which a weakly coupled job's
        // m > 0 can reach too
        bool acc = u < T || T == 0xFFFFFFFFu;
        if (J.weak && T == 0xFFFFFFFFu) {
            const int a = 2 * (ti >> 2) - (2 * D - 1);
            const int mm = a * J.den + ((ti & 2) ? P.w_self : -P.w_self) +
                           ((ti & 1) ? P.w_glue : -P.w_glue);
            acc = mm <= 0 || u != 0xFFFFFFFFu;
        }
        if (P.record) dE += ob ? 2 * (sf - gl) : 2 * (gl - sf);
        return (uint32_t)acc << sh;
    }

    __device__ __forceinline__ Edge edge_of(int t) const
    {
        const int lt = Lt(), rw = 4 * rowW(), repW = lt * rw, n = g.nrep;
        Edge e;
        e.t = t;
        e.n = t == 0 ? (lt - 1) * rw : (t == 1 ? (lt == 2 ? -rw : rw) : -rw);
        e.x = t == 0 ? rw : t == 1 ? -rw : (t == lt - 1 ? -(lt - 1) * rw : rw);
        e.g = t == 0 ? repW : t == 1 ? -repW : 0;
        e.gw = t == 0 ? -(n - 1) * repW : t == 1 ? (n - 1) * repW : 0;
        e.rw = t == 0 ? n - 1 : 0;
        return e;
    }

    // Bulk row, 2 <= t < L_t, all links full beta.  o: the word's position in
    // the other colour; own: in its own; up: byte offset of the t+1 row.
    __device__ __forceinline__ void bulk_row(A own_b, A oth, A own, A o, int up, const XShift& x,
                                             const uint4& ua, const uint4& ub) const
    {
        const uint32_t ow = ld(own_b, own, 1);
        uint32_t s = ld(oth, o - 4 * rowW(), 10) + ld(oth, o + up, 11) + ld(oth, o, 5) +
                     xjoin(ld(oth, o + x.a, 6), ld(oth, o + x.b, 6), x);
        if (D == 3) s += ld(oth, o + d_ym, 7) + ld(oth, o + d_yp, 8);
        uint32_t f = flips(s, ow, ua, ub);
        if (!FAST) f &= vmask;
        st(own_b, own, ow ^ f, 9);
    }

    // What the edge rows of a half-sweep share: row parity p, glue mask m
    // (nibbles with x < lg, empty for a row away from the cut) and the word's
    // first switched site jlo (x = 2 (8q + j) + p, g0 <= x < g1; 8 if none).
    struct Cut {
        uint32_t m;
        int jlo, p;
    };
    __device__ __forceinline__ Cut cut_of(const Edge& e, int c, const StepState& P) const
    {
        Cut k;
        k.p = (c + y + e.t) & 1;
        const bool cut = e.t < 2;
        k.m = cut ? glue_mask(P.lg, k.p) : 0u;
        k.jlo = cut && P.k >= 0 ? max(((J.g0 - k.p + 1) >> 1) - 8 * q, 0) : 8;
        return k;
    }

    // Edge row of replica r in one instruction stream for cut rows and others;
    // only the switched sites of a cut row take the per-site loop.
    __device__ __forceinline__ void edge_row(A own_b, A oth, int w4, const Edge& e, const Cut& k,
                                             int r, const XShift& x, const uint4& ua,
                                             const uint4& ub, const StepState& P, int& dE) const
    {
        const A o = oth + w4;
        const uint32_t own = ld(own_b, own_b + w4, 1);
        const uint32_t nrm = ld(oth, o + e.n, 2);
        const uint32_t self_w = ld(oth, o + e.x, 3);
        const uint32_t glue_w = ld(oth, o + e.x + (r == e.rw ? e.gw : e.g), 4);
        const uint32_t cross = (self_w & ~k.m) | (glue_w & k.m);
        uint32_t s = nrm + cross + ld(oth, o, 5) +
                     xjoin(ld(oth, o + x.a, 6), ld(oth, o + x.b, 6), x);
        if (D == 3) s += ld(oth, o + d_ym, 7) + ld(oth, o + d_yp, 8);
        uint32_t f = flips(s, own, ua, ub);
        if (k.jlo < 8) {
            const int jhi = min(((J.g1 - k.p + 1) >> 1) - 8 * q, 8);
#pragma unroll 1
            for (int jl = k.jlo; jl < jhi; ++jl)
                f = (f & ~(0xFu << (4 * jl))) |
                    switched_site(jl, own, self_w, glue_w, s,
                                  HALF ? word_of(ua, jl) : word8(ua, ub, jl), P, dE);
        }
        if (!FAST) f &= vmask;
        st(own_b, own_b + w4, own ^ f, 9);
    }

    // A replica's bulk rows, from word w4 (byte offset) and Philox product p0 on.
    // ODD: the slice step is odd, so the row parity alternates, starting with p.
    template <bool ODD>
    __device__ __forceinline__ void bulk_rows(A own_b, A oth, int w4, uint64_t p0, int p, XShift x,
                                              const Stream& st) const
    {
        const uint64_t dp = (uint64_t)kPhiloxM0 * (uint32_t)(step() * Ly() * G());
        const int stride = step() * rowW() * 4;
        A own = own_b + w4, o = oth + w4;
        auto row = [&](int up) {
            const uint4 ua = draw(p0, st);
            const uint4 ub = second(p0, st);
            bulk_row(own_b, oth, own, o, up, x, ua, ub);
            p0 += dp;
            own += stride;
            o += stride;
            if (ODD) x = xshift(p ^= 1);
        };
        int up = 4 * rowW();
        if constexpr (CLT > 0 && CTS > 2 && CLT % CTS == 0) {
            // as many rows for every slot, known at compile time: equal passes of at
            // most six (15 rows: three of five, 2D L = 64 scan 523 ms; 532 in fours
            // with a remainder, 529 in sevens)
            constexpr int N = CLT / CTS - 1;
            constexpr int PASS = N % 6 == 0 ? 6 : N % 5 == 0 ? 5 : N % 4 == 0 ? 4 : N % 3 == 0 ? 3 : 1;
#pragma unroll 1
            for (int h = 0; h < N / PASS; ++h) {
#pragma unroll
                for (int k = 0; k < PASS; ++k) row(up);
            }
        } else {
            // n_all rows that every slot has, four per pass and then singly,
            // so that a warp's slots do not diverge; then the last row, which
            // some slots lack and whose t + 1 row may wrap around
            int n = n_all;
#pragma unroll 1
            for (; n >= 4; n -= 4) {
#pragma unroll
                for (int i = 0; i < 4; ++i) row(up);
            }
#pragma unroll 1
            for (; n >= 0; --n) {
                if (n == 0) {
                    if (!has_last) break;
                    up = up_last;
                }
                row(up);
            }
        }
    }

    // The half-sweep of colour c.  With TS >= 3 slice steps slot t0 starts with
    // row t0 - 1 (slot 0 with L_t - 1): the two rows next to the cut and the row
    // whose t + 1 neighbour wraps around are all first rows, one instruction
    // stream for the whole team, and every other row is t0 - 1 + k TS with plain
    // time neighbours.  With TS <= 2 the cut rows t = 0, 1 come first, one per
    // slot or both, and the last bulk row wraps.  From TS = 2 on a thread has one
    // edge row per replica, whose geometry is `edge` (3D L = 16: 159.4 -> 154.9 ms;
    // short lattices, L_t = 2, L = 4 .. 40: 0.79 .. 0.88 of the time); TS = 1
    // recomputes that of its two rows.
    __device__ __forceinline__ void half_sweep(int c, uint32_t sweep, const StepState& P,
                                               int& dE) const
    {
        const int rw = rowW();
        const int lt = Lt();
        const A own_b = colour(c), oth = colour(c ^ 1);
        const int ts = step();
        if (t0 >= lt) return;   // a thread without sites
        const Stream st = stream(c, sweep);
        const bool one = ts >= 2;   // one edge row per replica, `edge`
        const Cut k0 = cut_of(edge, c, P);
        const XShift x0 = xshift(k0.p);
#pragma unroll 1
        for (int r = r0; r < g.nrep; r += RS) {
            const int wr = r * lt * rw + y * W() + q;   // word of slice 0
            const uint32_t cr = (uint32_t)((r * lt * Ly() + y) * G() + 2 * q);
            auto first = [&](const Edge& e, const Cut& k, const XShift& x) {
                const uint64_t p0 = (uint64_t)kPhiloxM0 * (cr + (uint32_t)(e.t * Ly() * G()));
                const uint4 ua = draw(p0, st);
                const uint4 ub = second(p0, st);
                edge_row(own_b, oth, 4 * (wr + e.t * rw), e, k, r, x, ua, ub, P, dE);
            };
            if (one) {
                first(edge, k0, x0);
            } else {
#pragma unroll 1
                for (int t = t0; t < 2; t += ts) {
                    const Edge e = edge_of(t);
                    const Cut k = cut_of(e, c, P);
                    first(e, k, xshift(k.p));
                }
            }
            const uint64_t p0 = (uint64_t)kPhiloxM0 * (cr + (uint32_t)(tb * Ly() * G()));
            const int w4 = 4 * (wr + tb * rw);
            const int p = (c + y + tb) & 1;
            if (CTS == 0 && (ts & 1)) bulk_rows<true>(own_b, oth, w4, p0, p, xshift(p), st);
            else bulk_rows<false>(own_b, oth, w4, p0, p, one ? x0 : xshift(p), st);
        }
    }

    // Loads a stored configuration (int8 +-1, natural order [r][t][y][x]) into
    // this thread's words: site j of word (c, R, q) has x = 2 (8q + j) + p.
    __device__ __forceinline__ void import_spins(const int8_t* src) const
    {
        const int rw = rowW();
        for (int c = 0; c < 2; ++c) {
            const A base = colour(c);
            for (int r = r0; r < g.nrep; r += RS) {
                int w = (r * g.Lt + t0) * rw + y * W() + q;
                for (int t = t0; t < g.Lt; t += TS, w += TS * rw) {
                    const int p = (c + t + y) & 1;
                    const long long row0 = ((long long)(r * g.Lt + t) * Ly() + y) * g.L;
                    uint32_t v = 0;
                    for (int j = 0; j < 8; ++j) {
                        const int x = 2 * (8 * q + j) + p;
                        if (x < g.L && src[row0 + x] < 0) v |= 1u << (4 * j);
                    }
                    st(base, base + 4 * w, v, 12);
                }
            }
        }
    }

    __device__ __forceinline__ void hot_start() const
    {
        const int rw = rowW();
        const uint32_t cstride = (uint32_t)(TS * Ly() * g.G);
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            const A base = colour(c);
            const uint32_t c3 = (uint32_t)c | c3base | (1u << 30);
#pragma unroll 1
            for (int r = r0; r < g.nrep; r += RS) {
                int w = (r * g.Lt + t0) * rw + y * W() + q;
                uint32_t c0 = (uint32_t)(((r * g.Lt + t0) * Ly() + y) * g.G + 2 * q);
#pragma unroll 1
                for (int t = t0; t < g.Lt; t += TS, w += TS * rw, c0 += cstride) {
                    const uint4 ua = philox_r0(c0, 0u, hi1, lo1, c3, K);
                    const uint4 ub = philox_r0(c0 + 1u, 0u, hi1, lo1, c3, K);
                    const uint32_t v = (ua.x >> 31) | ((ua.y >> 31) << 4) | ((ua.z >> 31) << 8) |
                                       ((ua.w >> 31) << 12) | ((ub.x >> 31) << 16) |
                                       ((ub.y >> 31) << 20) | ((ub.z >> 31) << 24) |
                                       ((ub.w >> 31) << 28);
                    st(base, base + 4 * w, v & vmask, 12);
                }
            }
        }
    }
};

struct CtaBarrier {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};
struct WarpBarrier {
    __device__ __forceinline__ void operator()() const { __syncwarp(); }
};

// The protocol's course through a trajectory's sweeps: thermalisation sweeps
// 0 .. n_therm - 1 at the start geometry (forward lambda = 0: x < g0 glued;
// reverse lambda = 1: x < g1 glued), then sweep i of step k is sweep n_therm +
// k n_sweep + i.  One loop runs both, so that the half-sweep's code exists once.
template <int D>
struct Course {
    const TeamJob& J;
    uint32_t s;      // global sweep index
    int k, left;     // step, sweeps left in it
    StepState P;

    __device__ __forceinline__ explicit Course(const TeamJob& J_) : J(J_)
    {
        const bool resume = J.k_begin > 0 || J.start_in;
        s = resume ? (uint32_t)J.n_therm + (uint32_t)J.k_begin * (uint32_t)J.n_sweep : 0u;
        k = J.k_begin - 1;
        left = resume ? 0 : J.n_therm;
        P = StepState{-1, J.dir > 0 ? J.g0 : J.g1, 0, 0, J.tcut, false};
    }
    // To the next sweep; false after the last one.
    __device__ __forceinline__ bool next()
    {
        if (left == 0) {
            if (++k >= J.k_end) return false;
            left = J.n_sweep;
            const int kp = k + 1 - active() * J.den;
            P.w_self = J.dir > 0 ? J.den - kp : kp;
            P.w_glue = J.dir > 0 ? kp : J.den - kp;
            P.k = k;
            P.lg = J.g0;
            P.tk = J.tcut + (size_t)k * (8 * D);
            P.record = true;
        }
        --left;
        return true;
    }
    // Protocol 2: only column y = active() moves at step k >= 0.
    __device__ __forceinline__ int active() const { return J.prot == 2 ? k / J.den : 0; }
    // The sweep's state for row y (protocol 2: the columns before the active one
    // sit at the end geometry, the ones after it at the start geometry).
    __device__ __forceinline__ StepState of_row(int y) const
    {
        StepState s = P;
        if (D == 3 && J.prot == 2 && P.k >= 0) {
            const int ya = active();
            if (y != ya) {
                s.k = -1;
                s.lg = (y < ya) == (J.dir > 0) ? J.g1 : J.g0;
            }
        }
        return s;
    }
};

// A trajectory whose team has a thread per word (2D, L = 16 and n L_t <= 32: one
// warp or less).  So few warps share an SM that nothing hides a half-sweep's
// latency but the warp itself, so each half-sweep draws the next one's
// Philox blocks and counts their thresholds (neither depends on spins) beside
// its own update, both colours' own words stay in registers, and everything of
// rounds 0 to 2 that does not depend on the sweep is computed once.
template <class Tr, class Bar>
__device__ __forceinline__ int run_rows(const Tr& tr, const Geom& g, const PhiloxKeys& K,
                                        const TeamJob& J, Bar bar)
{
    const int w = tr.r0 * g.Lt + tr.t0;   // one word per row
    const bool here = tr.t0 < g.Lt;
    const auto e = tr.edge_of(tr.t0);
    const int off_g = e.x + (tr.r0 == e.rw ? e.gw : e.g);
    const bool cut = here && tr.t0 < 2;
    uint32_t own[2] = {0u, 0u};
    // per colour and block: the counter entering round 2 but for its word 2,
    // and M0 times its word 0
    uint32_t c1[2][2], plo[2][2], phi[2][2], lop[2];
    int jlo[2], jhi[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        if (here) own[c] = tr.ld(tr.colour(c), tr.colour(c) + 4 * w, 1);
        const int p = (c + tr.t0) & 1;
        jlo[c] = cut ? max((J.g0 - p + 1) >> 1, 0) : 8;
        jhi[c] = min((J.g1 - p + 1) >> 1, 8);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const uint64_t p0 = (uint64_t)kPhiloxM0 * (uint32_t)(w * g.G + b);
            const uint64_t q1 = (uint64_t)kPhiloxM1 *
                                ((uint32_t)(p0 >> 32) ^ ((uint32_t)c | tr.c3base) ^ K.k1[0]);
            const uint64_t q0 =
                (uint64_t)kPhiloxM0 * ((uint32_t)(q1 >> 32) ^ tr.lo1 ^ K.k0[1]);
            c1[c][b] = (uint32_t)q1 ^ K.k0[2];
            plo[c][b] = (uint32_t)q0;
            phi[c][b] = (uint32_t)(q0 >> 32) ^ K.k1[2];
            lop[b] = (uint32_t)p0 ^ K.k1[1];
        }
    }
    auto draw = [&](uint32_t sweep, int c, uint4 u[2]) {
        const uint64_t q0 = (uint64_t)kPhiloxM0 * (tr.hi1 ^ sweep ^ K.k0[0]);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const uint64_t q1 = (uint64_t)kPhiloxM1 * ((uint32_t)(q0 >> 32) ^ lop[b]);
            u[b] = philox_from<3>((uint32_t)(q1 >> 32) ^ c1[c][b], (uint32_t)q1,
                                  phi[c][b] ^ (uint32_t)q0, plo[c][b], K);
        }
    };
    int dE = 0;
    Course<2> C(J);
    uint4 u[2];
    draw(C.s, 0, u);
    uint32_t n = count8<2>(u[0], u[1], J.tb);
    uint32_t m[2];
    int lg = -1;
    auto half = [&](int c) {
        const auto own_b = tr.colour(c), oth = tr.colour(c ^ 1), o = oth + 4 * w;
        uint32_t f = 0, nrm = 0, self_w = 0, glue_w = 0;
        if (here) {
            nrm = tr.ld(oth, o + e.n, 2);
            self_w = tr.ld(oth, o + e.x, 3);
            glue_w = tr.ld(oth, o + off_g, 4);
        }
        uint4 v[2];
        draw(c ? C.s + 1u : C.s, c ^ 1, v);
        const uint32_t nn = count8<2>(v[0], v[1], J.tb);
        const uint32_t ow = own[c], nx0 = own[c ^ 1];
        const int p = (c + tr.t0) & 1;
        const uint32_t s = nrm + ((self_w & ~m[c]) | (glue_w & m[c])) + nx0 +
                           __funnelshift_r(nx0, nx0, p ? 4 : 28);
        f = flips_of_counts<2>(s, ow, n);
        if (C.P.k >= 0) {
#pragma unroll 1
            for (int jl = jlo[c]; jl < jhi[c]; ++jl)
                f = (f & ~(0xFu << (4 * jl))) |
                    tr.switched_site(jl, ow, self_w, glue_w, s, word8(u[0], u[1], jl), C.P, dE);
        }
        own[c] = ow ^ f;
        if (here) tr.st(own_b, own_b + 4 * w, own[c], 9);
        u[0] = v[0];
        u[1] = v[1];
        n = nn;
        bar();
    };
#pragma unroll 1
    while (C.next()) {
        if (C.P.lg != lg) {
            lg = C.P.lg;
            m[0] = cut ? tr.glue_mask(lg, tr.t0 & 1) : 0u;
            m[1] = cut ? tr.glue_mask(lg, (tr.t0 + 1) & 1) : 0u;
        }
        half(0);
        C.P.record = false;
        half(1);
        ++C.s;
    }
    return dE;
}

// Runs one whole trajectory with the team's threads.  Every thread sharing the
// barrier calls it with the same job (trip counts match across teams); tid < 0
// marks a thread without sites.  Returns this thread's share of sum_k dE_k
// (the caller applies the direction's sign and, in protocol 2, the factor L_y
// that makes W = (beta/N) W_int).
// sin: the stored state to start from when J.k_begin > 0 or J.start_in (else unused).
// ROW: the team has a thread per word (run_rows).
template <int D, int KIND, bool PAIR, bool HBM, int CW, int CLY, bool ROW = false, int CLT = 0,
          int CTS = 0, class Bar>
__device__ __forceinline__ int run_trajectory(const Geom& g, const PhiloxKeys& K, const TeamJob& J,
                                              long long traj, uint32_t* S_team, const uint2* tab,
                                              int tid, int nthr, Bar bar,
                                              const int8_t* sin = nullptr)
{
    constexpr bool TAIL = KIND == kHalfTail;
    const Traj<D, KIND == kWhole, PAIR, HBM, CW, CLY, CLT, CTS, TAIL ? kWholeWords : kAllWords> tr(
        g, S_team, tab, J, K, (uint32_t)traj, tid, nthr);
    // rows that end in half a word: the half words have threads of their own
    const Traj<D, false, PAIR, HBM, CW, CLY, CLT, CTS, kTailWords> tail(g, S_team, tab, J, K,
                                                                       (uint32_t)traj, tid, nthr);
    if (J.k_begin > 0 || J.start_in) {
        if (tid >= 0) {
            tr.import_spins(sin);
            if (TAIL) tail.import_spins(sin);
        }
    } else {
        tr.hot_start();
        if (TAIL) tail.hot_start();
    }
    bar();
    if constexpr (ROW) {
        return run_rows(tr, g, K, J, bar);
    } else {
        int dE = 0;
        Course<D> C(J);
#pragma unroll 1
        while (C.next()) {
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
                tr.half_sweep(c, C.s, C.of_row(tr.y), dE);
                if (TAIL) tail.half_sweep(c, C.s, C.of_row(tail.y), dE);
                bar();
                C.P.record = false;
            }
            ++C.s;
        }
        return dE;
    }
}

// Writes a team's final configuration as int8 +-1 in the order [r][t][y][x].
template <int D>
__device__ __forceinline__ void export_spins(const Geom& g, const uint32_t* S_team, int8_t* dst,
                                             int tid, int nthr)
{
    const int V = g.nrep * g.Lt * g.Ly * g.L;
    for (int i = tid; i < V; i += nthr) {
        const int x = i % g.L;
        const int R = i / g.L;                      // (r, t, y) row
        int y = 0, trow = R;
        if (D == 3) { y = R % g.Ly; trow = R / g.Ly; }
        const int t = trow % g.Lt;
        const int c = (x + y + t) & 1;
        const int h = x >> 1;
        const long long wi = (long long)(c * g.NR + R) * g.GW + (h >> 3);
        const uint32_t word = in_bounds(wi, 2LL * g.NR * g.GW, 13) ? S_team[wi] : 0u;
        dst[i] = ((word >> (4 * (h & 7))) & 1u) ? (int8_t)-1 : (int8_t)1;
    }
}

// ly: L_y of the job's lattice (the number of switched columns).
__device__ __forceinline__ TeamJob team_job(const JobDesc& J, int ly)
{
    TeamJob t;
    t.l = __ldg(&J.l);
    t.n_step = __ldg(&J.n_step);
    t.n_sweep = __ldg(&J.n_sweep);
    t.n_therm = __ldg(&J.n_therm);
    t.dir = __ldg(&J.dir);
    t.prot = __ldg(&J.prot);
    t.k_begin = __ldg(&J.k_begin);
    t.k_end = __ldg(&J.k_end);
    t.start_in = __ldg(&J.start_in);
    t.g0 = __ldg(&J.g0);
    t.g1 = __ldg(&J.g1);
    t.den = t.prot == 2 ? t.n_step / ly : t.n_step;
    t.tcut = J.tcut;
    t.weak = __ldg(&J.weak) != 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) t.tb[a] = __ldg(&J.tb[a]);
    return t;
}

// This thread's team and team-local id under a launch shape (warp teams do
// not cross warps).  team = -1: no team.
__device__ __forceinline__ void team_of(const LaunchShape& sh, int* team, int* tid)
{
    const int x = (int)threadIdx.x;
    if (!sh.warp) {
        *team = 0;
        *tid = x;
        return;
    }
    const int per_warp = 32 / sh.team_threads;
    const int lane = x & 31;
    const int sub = lane / sh.team_threads;
    if (sub >= per_warp) {
        *team = -1;
        *tid = -1;
        return;
    }
    *team = (x >> 5) * per_warp + sub;
    *tid = lane - sub * sh.team_threads;
}

}  // namespace jz
