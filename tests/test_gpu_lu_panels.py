"""k_lu_solve with every panel width at sizes around the panel and the blocks of the substitution (the width is chosen by
the number of unknowns, and the narrowest needs more than 3200), several systems at a time: the kernel compiled
into a program of its own, residuals on the host.

Tolerance: Gaussian elimination with partial pivoting has a backward error below 8 N rho 2^-53 with a growth factor
rho below N^(2/3) for random matrices, so |A x - b| <= 8 N^(5/3) 2^-53 N max|A| max|x| for each element."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_01211_gb300", "csrc")
NVCC = next((p for p in ("/usr/local/cuda/bin/nvcc", shutil.which("nvcc")) if p and os.path.exists(p)), None)

MAIN = r"""
#include <cmath>
#include <complex>
#include <cstdio>
#include <vector>
#include "ng_setup.cuh"
typedef std::complex<double> C;
static unsigned long long state = 1911;
static double rnd() {
    state = state * 6364136223846793005ull + 1442695040888963407ull;
    return (double)(state >> 11) / 9007199254740992.0 - 0.5;
}
template <int PB>
static int check(int N, int nrhs) {
    const int nb = 3, ld = N + nrhs;
    std::vector<C> A((size_t)nb * N * ld), X(A.size());
    for (auto& x : A) x = C(rnd(), rnd());
    cplx* d;
    int *piv, *status, flags = 0;
    if (cudaMalloc(&d, sizeof(C) * A.size()) || cudaMalloc(&piv, sizeof(int) * nb * N) || cudaMalloc(&status, sizeof(int))) return 2;
    cudaMemcpy(d, A.data(), sizeof(C) * A.size(), cudaMemcpyHostToDevice);
    cudaMemset(status, 0, sizeof(int));
    const size_t smem = sizeof(cplx) * ((size_t)N * PB + NG_LU_TRI * nrhs);
    cudaFuncSetAttribute(k_lu_solve<PB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    dep_launch(k_lu_solve<PB>, nb, NG_LU_THREADS, smem, 0)(N, nrhs, d, piv, status);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    cudaMemcpy(X.data(), d, sizeof(C) * X.size(), cudaMemcpyDeviceToHost);
    cudaMemcpy(&flags, status, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(d); cudaFree(piv); cudaFree(status);
    if (flags) { printf("panel %d N %d: flags %d\n", PB, N, flags); return 1; }
    for (int b = 0; b < nb; ++b)
        for (int j = 0; j < nrhs; ++j) {
            double big = 0, worst = 0;
            for (int i = 0; i < N; ++i) big = std::max(big, std::abs(X[((size_t)b * N + i) * ld + N + j]));
            for (int r = 0; r < N; ++r) {
                C s = -A[((size_t)b * N + r) * ld + N + j];
                for (int i = 0; i < N; ++i) s += A[((size_t)b * N + r) * ld + i] * X[((size_t)b * N + i) * ld + N + j];
                worst = std::max(worst, std::abs(s));
            }
            const double tol = 8 * pow(N, 5.0 / 3.0) * pow(2, -53) * N * 0.7072 * big;
            if (!(worst <= tol)) { printf("panel %d N %d rhs %d: %g > %g\n", PB, N, j, worst, tol); return 1; }
        }
    return 0;
}
int main() {
    for (int N : {1, 2, 3, 8, 15, 16, 17, 31, 33, 100, 129})
        for (int nrhs : {1, 2, 5, 8})
            if (int e = check<2>(N, nrhs) | check<4>(N, nrhs) | check<8>(N, nrhs) | check<16>(N, nrhs)) return e;
    return 0;
}
"""


@pytest.mark.skipif(NVCC is None, reason="nvcc not found")
def test_every_panel_width(tmp_path):
    (tmp_path / "main.cu").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I", CSRC, str(tmp_path / "main.cu"),
                    "-o", exe], check=True, timeout=600)
    r = subprocess.run([exe], stdout=subprocess.PIPE, universal_newlines=True, timeout=300)
    assert r.returncode == 0, r.stdout
