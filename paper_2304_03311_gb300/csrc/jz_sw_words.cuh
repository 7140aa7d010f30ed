// jz_sw_words.cuh -- word arithmetic of the Swendsen-Wang kernel's grouped bond
// phase: 32 sites of a bit array at a time.  It compiles as plain C++ too, so
// that a CPU test can compare every word and direction of a lattice with the
// per-site form and see every index it reads.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define JZ_HD __host__ __device__ __forceinline__
#else
#define JZ_HD inline
#endif

namespace jz {

// Division by a fixed divisor d >= 1 for numerators n < 2^31 (Granlund and
// Montgomery, PLDI'94): with s = ceil(log2 d) and m = floor(2^32 (2^s - d) / d)
// + 1, n / d = (umulhi(m, n) + n) >> s.
struct FastDiv {
    uint32_t d, m, s;
};

inline FastDiv make_fastdiv(uint32_t d)
{
    uint32_t s = 0;
    while ((1ull << s) < d) ++s;
    const uint64_t m = (((1ull << s) - d) << 32) / d + 1;
    return FastDiv{d, (uint32_t)m, s};
}

JZ_HD uint32_t fdiv(uint32_t n, const FastDiv& f)
{
#ifdef __CUDA_ARCH__
    return (__umulhi(f.m, n) + n) >> f.s;
#else
    return ((uint32_t)(((uint64_t)f.m * n) >> 32) + n) >> f.s;
#endif
}

JZ_HD int mod(int a, const FastDiv& f) { return a - (int)(fdiv((uint32_t)a, f) * f.d); }

// The low word of hi:lo shifted right by s < 32.
JZ_HD uint32_t funnel_right(uint32_t lo, uint32_t hi, uint32_t s)
{
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, s);
#else
    return (uint32_t)(((((uint64_t)hi) << 32) | lo) >> s);
#endif
}

// Lowest and highest set bit of m != 0.
JZ_HD int first_bit(uint32_t m)
{
#ifdef __CUDA_ARCH__
    return __ffs((int)m) - 1;
#else
    return __builtin_ctz(m);
#endif
}
JZ_HD int last_bit(uint32_t m)
{
#ifdef __CUDA_ARCH__
    return 31 - __clz((int)m);
#else
    return 31 - __builtin_clz(m);
#endif
}

// Bits lo .. hi - 1 of a word, clipped to it.
JZ_HD uint32_t bit_range(int lo, int hi)
{
    lo = lo < 0 ? 0 : lo;
    hi = hi > 32 ? 32 : hi;
    if (lo >= hi) return 0u;
    return (hi == 32 ? 0xFFFFFFFFu : (1u << hi) - 1u) & ~((1u << lo) - 1u);
}

// The bits of a word whose sites' residues (the first one's: r) lie in [lo, hi)
// of a period.
JZ_HD uint32_t residue_bits(int r, int period, int lo, int hi)
{
    uint32_t m = 0;
    for (int b = -r; b < 32; b += period) m |= bit_range(b + lo, b + hi);
    return m;
}

// The wanted bits of o .. o + 31 of a bit array (the others are undefined).  Only
// words that hold wanted bits are read: the ones next to the array belong to
// others, who may be writing them.  Bits: has(i) says that bit i is inside the
// array (checked in bounds-checked builds, which skip the read otherwise), [w] is
// its word w.
template <class Bits>
JZ_HD uint32_t bits_at(const Bits& a, int o, uint32_t want)
{
    if (want == 0u || !a.has(o + first_bit(want)) || !a.has(o + last_bit(want))) return 0u;
    const int w = o >> 5;
    const uint32_t s = (uint32_t)o & 31u, low = 0xFFFFFFFFu >> s;   // low: bits of word w
    const uint32_t lo = (want & low) ? a[w] : 0u;
    const uint32_t hi = (want & ~low) ? a[w + 1] : 0u;
    return funnel_right(lo, hi, s);
}

// The bits of the valid sites of a word W (its first site: base) that equal their
// neighbour at + o, or, for the sites `wraps` of them, at + o - wrap.
template <class Bits>
JZ_HD uint32_t equal_bits(const Bits& a, uint32_t W, int base, uint32_t valid, uint32_t wraps,
                          int o, int wrap)
{
    const uint32_t inner = valid & ~wraps;
    const uint32_t nb = (bits_at(a, base + o, inner) & inner) |
                        (bits_at(a, base + o - wrap, wraps) & wraps);
    return ~(W ^ nb) & valid;
}

// What a lane needs of word q: its first site, the valid bits, and the bits of
// the sites whose +x, +t and +y neighbours wrap around.  G: a lattice of V sites in
// replicas of VR, slices of SL and rows of L sites, with divisors dL, dSL, dVR.
struct WordPos {
    int base;
    uint32_t valid, x_end, t_end, y_end;
};

template <int D, class G>
JZ_HD WordPos word_pos(const G& g, int q)
{
    WordPos p;
    p.base = 32 * q;
    p.valid = bit_range(0, g.V - p.base);
    p.x_end = residue_bits(mod(p.base, g.dL), g.L, g.L - 1, g.L) & p.valid;
    p.t_end = residue_bits(mod(p.base, g.dVR), g.VR, g.VR - g.SL, g.VR) & p.valid;
    p.y_end = D == 3 ? residue_bits(mod(p.base, g.dSL), g.SL, g.SL - g.L, g.SL) & p.valid : 0u;
    return p;
}

}  // namespace jz
