"""The key of the pivot searches, compiled for the host (CPU only): finite magnitudes in their order, infinities
above them, and a NaN of either sign below zero, so that it never replaces a row."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1911_01211_gb300", "csrc")
NVCC = next((p for p in ("/usr/local/cuda/bin/nvcc", shutil.which("nvcc")) if p and os.path.exists(p)), None)

MAIN = r"""
#include <cmath>
#include <cstdio>
#include "ng_common.cuh"
int main() {
    const double up = NAN, down = copysign(NAN, -1.0), inf = INFINITY;
    const double row[] = {0.0, 1e-320, 1e-200, 1e-100, 0.5, 1.0, -1.0000001, 3.0, -1e100, 1e154, -inf};
    long long last = -1;
    for (double x : row) {
        const long long k = pivot_key(make_double2(x, 0.0));
        if (k < last || k < 0 || pivot_key(make_double2(0.0, -x)) != k) { printf("%g out of order\n", x); return 1; }
        last = k;
    }
    if (pivot_key(make_double2(0.0, -0.0)) != 0) { printf("zero\n"); return 1; }
    for (double bad : {up, down})
        for (double x : {0.0, 1.0, inf, bad})
            if (pivot_key(make_double2(bad, x)) != -1 || pivot_key(make_double2(x, bad)) != -1) { printf("NaN\n"); return 1; }
    return 0;
}
"""


@pytest.mark.skipif(NVCC is None, reason="nvcc not found")
def test_key_orders_magnitudes_and_rejects_nan(tmp_path):
    (tmp_path / "main.cu").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([NVCC, "-std=c++17", "-I", CSRC, str(tmp_path / "main.cu"), "-o", exe], check=True, timeout=300)
    r = subprocess.run([exe], stdout=subprocess.PIPE, universal_newlines=True, timeout=300)
    assert r.returncode == 0, r.stdout


def test_no_search_starts_outside_the_matrix():
    """The searches compare keys from -1 on and begin with a row of the matrix; with row N as their beginning a column of
    NaN (the sign bit set, CUDA's own pattern) left row N, the next problem's, as the pivot."""
    for name in ("ng_step.cuh", "ng_setup.cuh"):
        src = open(os.path.join(CSRC, name)).read()
        assert "__double_as_longlong(cabs2" not in src
        assert "int p = N;" not in src and "int bi = N;" not in src
