"""The Swendsen-Wang kernels for states beyond shared memory, as the assembler reports
them: no spills, and registers that let the CTAs per SM share it that a wave of such
states counts on (kHbmCtas2d, kHbmCtas3d), or two for 3D launches that two per SM
hold."""
import os
import re
import shutil
import subprocess

import pytest

from conftest import ROOT

NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
CSRC = os.path.join(ROOT, "paper_2304_03311_gb300", "csrc")


def test_hbm_variants_fit_their_waves(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    r = subprocess.run([NVCC, "-c", os.path.join(CSRC, "jz_sw.cu"), "-o", str(tmp_path / "sw.o"),
                        "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I",
                        os.path.join(ROOT, "include"), "-Xptxas", "-v"],
                       capture_output=True, text=True, check=True)
    src = open(os.path.join(CSRC, "jz_sw.cu")).read()
    wave = {d: int(re.search(r"kHbmCtas%dd = (\d)" % d, src).group(1)) for d in (2, 3)}
    seen = []
    # sw_kernel<D, HBM, GROUP, minimum CTAs per SM>
    for m in re.finditer(r"sw_kernelILi(\d)ELb(\d)ELb\d+ELi(\d+)E.*?(\d+) bytes spill stores, "
                         r"(\d+) bytes spill loads.*?Used (\d+) registers", r.stderr, re.S):
        d, hbm, ctas, st, ld, regs = map(int, m.groups())
        assert (st, ld) == (0, 0), m.group(0)
        if hbm:
            threads = 512 if d == 3 else 256
            need = 2 if ctas == 2 else wave[d]
            assert -(-regs // 8) * 8 * threads * need <= 65536, m.group(0)
            seen.append((d, need))
    assert sorted(seen) == [(2, wave[2]), (3, 2), (3, wave[3])], seen
