"""spread_smem (csrc/sd_internal.h): the shared memory it asks for lets exactly an even share of CTAs
onto an SM, static shared memory and the system's 1 KB a CTA included, or is what the kernel needs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include <cstdio>
#include "sd_internal.h"
int main() {
    const int sms = 152, sm = 228 * 1024;
    int bad = 0;
    for (int stat = 0; stat <= 40960; stat += 128)
        for (int need = 0; need <= 65536; need += 8192)
            for (int grid = 1; grid <= 20 * sms; grid += 37) {
                const int occ = sm / (need + stat + 1024), per = (grid + sms - 1) / sms;
                const size_t d = sd::spread_smem(sms, grid, occ, need, 227 * 1024 - stat);
                const int fit = sm / static_cast<int>(d + stat + 1024);
                // never less than needed or more than allowed; an even share fits (all that fit, if it does not)
                if (d < static_cast<size_t>(need) || d + stat > 227 * 1024 || fit != (per < occ ? per : occ)) {
                    if (++bad < 5) printf("static %d need %d grid %d: %zu, %d fit, share %d of %d\n", stat, need, grid, d, fit, per, occ);
                }
            }
    return bad != 0;
}
'''


def test_spread_smem_lets_an_even_share_fit(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(SRC)
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "paper_1205_6333_gb300", "csrc"), str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
