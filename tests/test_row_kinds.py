"""How a team works on rows that end in half a word (csrc/jz_device.cuh, row_kind):
half words on threads of their own where the half-sweep gets shorter by it, all words
in one pass where both ways leave a thread one row per pass.  Host code only."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
RAGGED, WHOLE, HALF_TAIL = 0, 1, 2
# d, L, L_t, team threads -> kind
CASES = [
    (3, 18, 2, 72, RAGGED), (3, 24, 2, 96, RAGGED), (3, 18, 4, 144, RAGGED),
    (3, 20, 6, 240, RAGGED), (3, 24, 4, 192, RAGGED),
    (3, 24, 96, 192, HALF_TAIL), (3, 24, 24, 192, HALF_TAIL), (3, 20, 20, 120, HALF_TAIL),
    (3, 18, 2, 36, HALF_TAIL),                              # two rows per thread in one pass
    (2, 8, 8, 16, HALF_TAIL), (2, 2, 2, 4, HALF_TAIL),
    (3, 36, 16, 432, HALF_TAIL), (3, 40, 20, 480, HALF_TAIL),   # throughput counts
    (3, 8, 8, 32, HALF_TAIL),                               # half words only: one pass
    (2, 64, 64, 32, WHOLE), (3, 28, 28, 112, RAGGED),       # none, and five to seven sites
]

DRIVER = r"""
#include <cstdio>
#include <cuda_runtime.h>
#include "jz_device.cuh"
int main()
{
    int d, L, Lt, thr;
    while (std::scanf("%d %d %d %d", &d, &L, &Lt, &thr) == 4) {
        const int Ly = d == 3 ? L : 1, Lh = L / 2;
        const jz::Geom g{L, Lt, Ly, Lh, (Lh + 3) / 4, (Lh + 7) / 8, 2, 2 * Lt * Ly};
        std::printf("%d\n", (int)jz::row_kind(g, jz::LaunchShape{thr, 1, thr, 0}));
    }
}
"""


@pytest.fixture(scope="module")
def kinds(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("kinds")
    src, exe = d / "kinds.cu", d / "kinds"
    src.write_text(DRIVER)
    subprocess.run([NVCC, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_2304_03311_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    text = "".join("%d %d %d %d\n" % c[:4] for c in CASES)
    r = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True)
    return dict(zip((c[:4] for c in CASES), map(int, r.stdout.split())))


@pytest.mark.parametrize("case", CASES, ids=lambda c: "d%dL%dLt%dthr%d" % c[:4])
def test_row_kind(kinds, case):
    assert kinds[case[:4]] == case[4]
