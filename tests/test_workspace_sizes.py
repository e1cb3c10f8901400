"""Sizes of workspaces that are allocated for a run's last step and used by every step before it, from the
functions the library uses, compiled for the host (CPU only)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1911_01211_gb300", "csrc")
NVCC = next((p for p in ("/usr/local/cuda/bin/nvcc", shutil.which("nvcc")) if p and os.path.exists(p)), None)

MAIN = r"""
#include <cstdio>
#include "ng_histu.h"
// every step's parts of one problem's workspace lie behind one another and inside the bytes of any later step
int main() {
    for (int D = 1; D <= 8; D *= 2)
        for (int T : {33, 100, 300, 1000}) {
            int64_t most = 0;
            for (int n = 1; n <= 4000; ++n) {
                HistUGeo q;
                histu_geo(D, T, n, q);
                int64_t el = q.part;
                for (int s = 0; s < NGU_SETS; ++s) {
                    if (q.part + q.poff[s] * 16 < el || q.kt[s] > 256 ||
                        q.task0[s + 1] - q.task0[s] != q.free_[s] / NGU_M * q.chunks[s]) {
                        printf("layout D %d T %d n %d set %d\n", D, T, n, s);
                        return 1;
                    }
                    el = q.part + (q.poff[s] + (int64_t)q.free_[s] * q.chunks[s] * D) * 16;
                }
                if (el > q.bytes || q.bytes < most) {
                    printf("D %d T %d n %d: %lld bytes used, %lld allotted, %lld by an earlier step\n", D, T, n, (long long)el,
                           (long long)q.bytes, (long long)most);
                    return 1;
                }
                most = q.bytes;
            }
        }
    return 0;
}
"""


@pytest.mark.skipif(NVCC is None, reason="nvcc not found")
def test_uneven_digit_workspace_grows_with_the_step(tmp_path):
    (tmp_path / "main.cu").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([NVCC, "-std=c++17", "-I", CSRC, str(tmp_path / "main.cu"), "-o", exe], check=True, timeout=300)
    r = subprocess.run([exe], stdout=subprocess.PIPE, universal_newlines=True, timeout=300)
    assert r.returncode == 0, r.stdout
