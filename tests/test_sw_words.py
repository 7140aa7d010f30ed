"""The Swendsen-Wang kernel's word arithmetic (csrc/jz_sw_words.cuh) compiled as
plain C++: for every word and direction of small lattices, rows, slices and
replicas that straddle words among them, the bits of sites equal to their +x, +t
and +y neighbours must be those of the per-site form, and no word outside the bit
array may be read (the words next to it belong to others, who write them in the
same phase)."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "jz_sw_words.cuh"

struct Bits {   // records every index outside the array
    const std::vector<uint32_t>& w;
    int V;
    long* bad;
    bool has(int i) const { return i >= 0 && i < V ? true : (++*bad, false); }
    uint32_t operator[](int q) const
    {
        if (q >= 0 && q < (int)w.size()) return w[q];
        ++*bad;
        return 0u;
    }
};
struct Geo {
    int V, VR, SL, L;
    jz::FastDiv dL, dSL, dVR;
};

template <int D>
long check(int L, int Lt, int n)
{
    const int SL = D == 3 ? L * L : L, VR = Lt * SL, V = n * VR;
    const Geo g{V, VR, SL, L, jz::make_fastdiv(L), jz::make_fastdiv(SL), jz::make_fastdiv(VR)};
    std::vector<uint32_t> sp((V + 31) / 32, 0u);
    std::vector<int> s(V);
    for (int i = 0; i < V; ++i) {
        s[i] = rand() & 1;
        sp[i >> 5] |= (uint32_t)s[i] << (i & 31);
    }
    long bad = 0;
    const Bits bits{sp, V, &bad};
    for (int q = 0; q < (int)sp.size(); ++q) {
        const jz::WordPos p = jz::word_pos<D>(g, q);
        const uint32_t x = jz::equal_bits(bits, sp[q], p.base, p.valid, p.x_end, 1, L);
        const uint32_t t = jz::equal_bits(bits, sp[q], p.base, p.valid, p.t_end, SL, VR);
        const uint32_t y =
            D == 3 ? jz::equal_bits(bits, sp[q], p.base, p.valid, p.y_end, L, SL) : 0u;
        uint32_t ex = 0, et = 0, ey = 0;
        for (int j = 0; j < 32 && 32 * q + j < V; ++j) {
            const int i = 32 * q + j, r = i / VR, tt = i % VR / SL, yy = i % SL / L, xx = i % L;
            ex |= (uint32_t)(s[i] == s[i - xx + (xx + 1) % L]) << j;
            et |= (uint32_t)(s[i] == s[r * VR + (tt + 1) % Lt * SL + i % SL]) << j;
            if (D == 3) ey |= (uint32_t)(s[i] == s[i - yy * L + (yy + 1) % L * L]) << j;
        }
        bad += (x != ex) + (t != et) + (y != ey);
    }
    if (bad) std::printf("%dD L = %d, L_t = %d, n = %d: %ld\n", D, L, Lt, n, bad);
    return bad;
}

int main()
{
    long bad = 0;
    for (int n : {2, 3, 8})
        for (int Lt : {2, 4, 6, 14, 32})
            for (int L : {2, 4, 6, 8, 10, 14, 16, 20, 22, 30, 32, 34, 50, 64, 70}) {
                bad += check<2>(L, Lt, n);
                if (L <= 16) bad += check<3>(L, Lt, n);
            }
    return bad != 0;
}
"""


def test_words_match_sites_and_stay_inside(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not found")
    src, exe = tmp_path / "words.cpp", tmp_path / "words"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I",
                    os.path.join(ROOT, "paper_2304_03311_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
