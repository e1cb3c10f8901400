// Setup kernels of libng: free Green's functions, the Matsubara solve and the start-up.
#pragma once

#include "ng_step.cuh"
#include "ng_stepsplit.cuh"

// ----------------------------------------------------------------------------------------
// Hermitian eigen-decomposition of a small D x D matrix by cyclic Jacobi rotations
// (Jacobi 1846; complex form as in Golub & Van Loan, Sec. 8.5).  eps = R diag(e) R^dagger.
// ----------------------------------------------------------------------------------------
template <int D>
__device__ void herm_eig(Mat<D> A, double e[D], Mat<D>& R) {
    R = meye<D>(cr(1.0));
    for (int sweep = 0; sweep < 30; ++sweep) {
        double off = 0.0;
        for (int p = 0; p < D; ++p)
            for (int q = p + 1; q < D; ++q) off += cabs2(A.v[p][q]);
        if (off < 1e-300) break;
        for (int p = 0; p < D; ++p)
            for (int q = p + 1; q < D; ++q) {
                double apq = sqrt(cabs2(A.v[p][q]));
                if (apq < 1e-300) continue;
                // phase so that the rotated element is real: A_pq = |A_pq| e^{i phi}
                cplx ph = make_double2(A.v[p][q].x / apq, A.v[p][q].y / apq);
                double app = A.v[p][p].x, aqq = A.v[q][q].x;
                double theta = 0.5 * atan2(2.0 * apq, aqq - app);
                double c = cos(theta), s = sin(theta);
                // unitary J acting on columns p, q: col_p' = c col_p - s conj(ph) col_q ... built as
                // J = [[c, s ph], [-s conj(ph), c]] in the (p, q) plane
                cplx jpp = cr(c), jpq = cscal(s, ph), jqp = cscal(-s, cconj(ph)), jqq = cr(c);
                // A <- J^dagger A J
                for (int r = 0; r < D; ++r) {  // A J (columns)
                    cplx arp = A.v[r][p], arq = A.v[r][q];
                    A.v[r][p] = cadd(cmul(arp, jpp), cmul(arq, jqp));
                    A.v[r][q] = cadd(cmul(arp, jpq), cmul(arq, jqq));
                    cplx rrp = R.v[r][p], rrq = R.v[r][q];
                    R.v[r][p] = cadd(cmul(rrp, jpp), cmul(rrq, jqp));
                    R.v[r][q] = cadd(cmul(rrp, jpq), cmul(rrq, jqq));
                }
                for (int r = 0; r < D; ++r) {  // J^dagger (rows)
                    cplx apr = A.v[p][r], aqr = A.v[q][r];
                    A.v[p][r] = cadd(cmul(cconj(jpp), apr), cmul(cconj(jqp), aqr));
                    A.v[q][r] = cadd(cmul(cconj(jpq), apr), cmul(cconj(jqq), aqr));
                }
            }
    }
    for (int a = 0; a < D; ++a) e[a] = A.v[a][a].x;
}

// (1 + xi f(e)) e^{-e tau} and f(e) e^{e tau} for fermions (xi = -1), overflow-safe
__device__ __forceinline__ void fermi_terms(double e, double beta, double tau, double* gm, double* gtv) {
    if (e >= 0.0) {
        double x = exp(-beta * e);
        *gm = exp(-e * tau) / (1.0 + x);
        *gtv = x / (1.0 + x) * exp(e * tau);
    } else {
        double x = exp(beta * e);
        *gm = exp(e * (beta - tau)) / (1.0 + x);
        *gtv = exp(e * tau) / (1.0 + x);
    }
}

// ----------------------------------------------------------------------------------------
// free Green's function of constant eps (Eq. G0_free), times `scale`; one thread per
// (element, problem).  eps_dev: [nb][D][D].
// ----------------------------------------------------------------------------------------
template <int D>
__global__ void k_free_gf(Grid g, HermV G, const cplx* eps_dev, double scale) {
    dep_wait();
    const int64_t nel_tri = tri(g.nt + 1);
    const int64_t nel_tv = (int64_t)(g.nt + 1) * (g.ntau + 1);
    const int64_t nel = (g.ntau + 1) + 2 * nel_tri + nel_tv;
    const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= nel * g.nb) return;
    const int kb = (int)(item % g.nb);
    int64_t e = item / g.nb;
    Mat<D> E;
    for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b) E.v[a][b] = eps_dev[(kb * D + a) * D + b];
    double ev[D];
    Mat<D> R;
    herm_eig<D>(E, ev, R);
    for (int a = 0; a < D; ++a) ev[a] -= g.mu;
    Mat<D> Rd = mdag<D>(R);
    auto sandwich = [&](const cplx* dg) {  // R diag(dg) R^dagger
        Mat<D> x;
        for (int a = 0; a < D; ++a)
            for (int b = 0; b < D; ++b) {
                cplx s = cz();
                for (int c = 0; c < D; ++c) s = cadd(s, cmul(cmul(R.v[a][c], dg[c]), Rd.v[c][b]));
                x.v[a][b] = s;
            }
        return x;
    };
    cplx dg[D];
    const double xi = (double)g.sig;
    if (e < g.ntau + 1) {  // mat: -R diag{(1 + xi f) e^{-e tau}} R^dagger
        const int m = (int)e;
        for (int c = 0; c < D; ++c) {
            double gm, gt;
            fermi_terms(ev[c], g.beta, m * g.htau, &gm, &gt);
            dg[c] = cr(-gm * scale);
        }
        st<D>(G.mat, m, kb, sandwich(dg));
        return;
    }
    e -= g.ntau + 1;
    if (e < 2 * nel_tri) {
        const bool isret = e < nel_tri;
        if (!isret) e -= nel_tri;
        // decode row n and column j of the packed triangle
        int n = (int)((sqrt(8.0 * (double)e + 1.0) - 1.0) * 0.5);
        while (tri(n + 1) <= e) ++n;
        while (tri(n) > e) --n;
        const int j = (int)(e - tri(n));
        const double dt = (n - j) * g.h;
        for (int c = 0; c < D; ++c) {
            double s, co;
            sincos(ev[c] * dt, &s, &co);
            if (isret) {
                dg[c] = cscal(scale, make_double2(-s, -co));    // -i e^{-i e dt}
            } else {
                double f = 0.5 * (1.0 - tanh(0.5 * g.beta * ev[c]));
                // G^<(j,n) = -xi i f e^{-i e (t_j - t_n)} = -xi i f e^{+i e dt}
                dg[c] = cscal(-xi * f * scale, make_double2(-s, co));
            }
        }
        st<D>(isret ? G.ret : G.les, e, kb, sandwich(dg));
        return;
    }
    e -= 2 * nel_tri;
    const int n = (int)(e / (g.ntau + 1)), m = (int)(e % (g.ntau + 1));
    for (int c = 0; c < D; ++c) {  // -i xi f e^{-i e t} e^{e tau}
        double gm, gt, s, co;
        fermi_terms(ev[c], g.beta, m * g.htau, &gm, &gt);
        sincos(ev[c] * n * g.h, &s, &co);
        cplx ph = make_double2(co, -s);
        dg[c] = cscal(xi * gt * scale, cmulmi(ph));  // -i xi f e^{e tau} e^{-i e t}
    }
    st<D>(G.tv, e, kb, sandwich(dg));
}

// ----------------------------------------------------------------------------------------
// Matsubara solve (Sec. "Matsubara"): g^M, K = [g * Sigma]^M, dense operator, LU.
// workspace layout per problem kb: gM[(T+1)][D][D], K[(T+1)][D][D], A[N][N+D] (augmented
// row-major, N = (T+1) D).
// ----------------------------------------------------------------------------------------
template <int D>
__global__ void k_mat_g(Grid g, FuncV eps, cplx* ws_g) {
    dep_wait();
    const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= (int64_t)(g.ntau + 1) * g.nb) return;
    const int kb = (int)(item % g.nb), m = (int)(item / g.nb);
    Mat<D> E = ldf<D>(eps, -1, kb);
    double ev[D];
    Mat<D> R;
    herm_eig<D>(E, ev, R);
    Mat<D> x;
    for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b) {
            cplx s = cz();
            for (int c = 0; c < D; ++c) {
                double gm, gt;
                fermi_terms(ev[c] - g.mu, g.beta, m * g.htau, &gm, &gt);
                s = cadd(s, cscal(-gm, cmul(R.v[a][c], cconj(R.v[b][c]))));
            }
            x.v[a][b] = s;
        }
    cplx* dst = ws_g + ((int64_t)kb * (g.ntau + 1) + m) * D * D;
    for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b) dst[a * D + b] = x.v[a][b];
}

// Matsubara convolution C^M_1[A,1,B](m) + C^M_2[A,1,B](m) (Eqs. cm1, cm2) with A taken from a
// per-problem workspace array and B from a herm component.
template <int D>
__device__ Mat<D> cmat_ws_comp(const NgWeights& W, const Grid& g, const cplx* Aws, const Comp& B, int m, int kb) {
    const int k = W.k, T = g.ntau;
    const double xi = (double)g.sig;
    auto A = [&](int i) {
        Mat<D> r;
        for (int a = 0; a < D; ++a)
            for (int b = 0; b < D; ++b) r.v[a][b] = Aws[i * D * D + a * D + b];
        return r;
    };
    Mat<D> c1 = mzero<D>(), c2 = mzero<D>();
    if (m <= k) {
        for (int j = 0; j <= k; ++j)
            for (int l = 0; l <= k; ++l) mfma<D>(c1, mscal<D>(W.R[m][j][l], A(j)), ld<D>(B, l, kb));
    } else {
        greg_for(W, m, m, [&](int l, double w) { mfma<D>(c1, mscal<D>(w, A(m - l)), ld<D>(B, l, kb)); });
    }
    if (m >= T - k) {
        for (int j = 0; j <= k; ++j)
            for (int l = 0; l <= k; ++l) mfma<D>(c2, mscal<D>(W.R[T - m][j][l], A(T - j)), ld<D>(B, T - l, kb));
    } else {
        greg_for(W, T - m, T - m, [&](int l, double w) { mfma<D>(c2, mscal<D>(w, A(T - l)), ld<D>(B, m + l, kb)); });
    }
    return mscal<D>(g.htau, madd<D>(c1, mscal<D>(xi, c2)));
}

// this lane's share of the terms of cmat_ws_comp
template <int D>
__device__ Mat<D> cmat_ws_comp_part(const NgWeights& W, const Grid& g, const cplx* Aws, const Comp& B, int m, int kb, int lane) {
    const int k = W.k, T = g.ntau, kk = (k + 1) * (k + 1);
    auto A = [&](int i) {
        Mat<D> r;
        for (int a = 0; a < D; ++a)
            for (int b = 0; b < D; ++b) r.v[a][b] = Aws[i * D * D + a * D + b];
        return r;
    };
    Mat<D> c1 = mzero<D>(), c2 = mzero<D>();
    if (m <= k) {
        for (int i = lane; i < kk; i += 32)
            mfma<D>(c1, mscal<D>(W.R[m][i / (k + 1)][i % (k + 1)], A(i / (k + 1))), ld<D>(B, i % (k + 1), kb));
    } else {
        greg_for_lanes(W, m, m, lane, [&](int l, double w) { mfma<D>(c1, mscal<D>(w, A(m - l)), ld<D>(B, l, kb)); });
    }
    if (m >= T - k) {
        for (int i = lane; i < kk; i += 32)
            mfma<D>(c2, mscal<D>(W.R[T - m][i / (k + 1)][i % (k + 1)], A(T - i / (k + 1))), ld<D>(B, T - i % (k + 1), kb));
    } else {
        greg_for_lanes(W, T - m, T - m, lane, [&](int l, double w) { mfma<D>(c2, mscal<D>(w, A(T - l)), ld<D>(B, m + l, kb)); });
    }
    return mscal<D>(g.htau, madd<D>(c1, mscal<D>((double)g.sig, c2)));
}
// sum over the warp's lanes, on every lane
template <int D>
__device__ __forceinline__ Mat<D> warp_sum_all(Mat<D> x) {
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = 0; b < D; ++b)
            for (int o = 16; o > 0; o >>= 1) {
                x.v[a][b].x += __shfl_xor_sync(0xffffffffu, x.v[a][b].x, o);
                x.v[a][b].y += __shfl_xor_sync(0xffffffffu, x.v[a][b].y, o);
            }
    return x;
}

template <int D>
__global__ void k_mat_K(Grid g, HermV S, const cplx* ws_g, cplx* ws_K) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= (int64_t)(g.ntau + 1) * g.nb) return;
    const int kb = (int)(item % g.nb), m = (int)(item / g.nb);
    Mat<D> K = cmat_ws_comp<D>(W, g, ws_g + (int64_t)kb * (g.ntau + 1) * D * D, S.mat, m, kb);
    cplx* dst = ws_K + ((int64_t)kb * (g.ntau + 1) + m) * D * D;
    for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b) dst[a * D + b] = K.v[a][b];
}

// Augmented matrix [I - A | g] of the linear map X -> C^M_1[K,1,X] + C^M_2[K,1,X]; one
// thread per (problem, block row m, block column c).
template <int D>
__global__ void k_mat_assemble(Grid g, const cplx* ws_g, const cplx* ws_K, cplx* ws_A) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int T = g.ntau, k = W.k;
    const int N = (T + 1) * D, ldA = N + D;
    const int64_t nblk = (int64_t)(T + 1) * (T + 2);
    const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= nblk * g.nb) return;
    const int kb = (int)(item / nblk);
    const int64_t r = item % nblk;
    const int m = (int)(r / (T + 2)), c = (int)(r % (T + 2));
    const cplx* K = ws_K + (int64_t)kb * (T + 1) * D * D;
    cplx* A = ws_A + (int64_t)kb * N * ldA;
    auto Kb = [&](int i) {
        Mat<D> x;
        for (int a = 0; a < D; ++a)
            for (int b = 0; b < D; ++b) x.v[a][b] = K[i * D * D + a * D + b];
        return x;
    };
    if (c == T + 1) {  // right-hand side g^M(tau_m)
        const cplx* gg = ws_g + ((int64_t)kb * (T + 1) + m) * D * D;
        for (int a = 0; a < D; ++a)
            for (int b = 0; b < D; ++b) A[(int64_t)(m * D + a) * ldA + N + b] = gg[a * D + b];
        return;
    }
    const double xi = (double)g.sig;
    Mat<D> blk = mzero<D>();
    if (m <= k) {
        if (c <= k)
            for (int j = 0; j <= k; ++j) blk = madd<D>(blk, mscal<D>(W.R[m][j][c], Kb(j)));
    } else if (c <= m) {
        blk = madd<D>(blk, mscal<D>(gw(W, m, c), Kb(m - c)));
    }
    if (m >= T - k) {
        if (c >= T - k)
            for (int j = 0; j <= k; ++j) blk = madd<D>(blk, mscal<D>(W.R[T - m][j][T - c] * xi, Kb(T - j)));
    } else if (c >= m) {
        blk = madd<D>(blk, mscal<D>(gw(W, T - m, c - m) * xi, Kb(T - (c - m))));
    }
    blk = mscal<D>(-g.htau, blk);
    if (c == m)
        for (int a = 0; a < D; ++a) blk.v[a][a].x += 1.0;
    for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b) A[(int64_t)(m * D + a) * ldA + c * D + b] = blk.v[a][b];
}

// ----------------------------------------------------------------------------------------
// Dense solves of the Matsubara systems.  Batches: LU, one block per problem (k_lu_solve,
// k_lu_resolve).  A few problems: the inverse by Gauss-Jordan elimination over the whole GPU, or for larger
// systems LU with the updates over the whole GPU (k_lu_col, k_lu_rank1, k_lu_backsub).
// ----------------------------------------------------------------------------------------
#define NG_LU_THREADS 512

// x_r for the W rows of a triangular block, lane (r, column) of one warp; A at the block's first element.
// Lanes take the (row, right-hand side) pairs in turn; unit lower (FWD) or upper triangle.
#define NG_LU_TRI 16
#define NG_LU_STAGE 1024
template <bool FWD>
__device__ void lu_tri_block(const cplx* A, int ld, int w, cplx* B, int ldb, int nrhs, int lane) {
    const int r = lane & (NG_LU_TRI - 1);
    cplx inv = cz();
    if (!FWD && r < w) inv = cinv(A[(int64_t)r * ld + r]);
    for (int j0 = 0; j0 < nrhs; j0 += 2) {   // two right-hand sides per pass: lanes 0..15, 16..31
        const int j = j0 + (lane >> 4);
        cplx x = (r < w && j < nrhs) ? B[r * ldb + j] : cz();
        for (int q = 0; q < w; ++q) {
            const int c = FWD ? q : w - 1 - q;
            if (!FWD && r == c) x = cmul(x, inv);
            cplx xc;
            xc.x = __shfl_sync(0xffffffffu, x.x, (lane & 16) + c);
            xc.y = __shfl_sync(0xffffffffu, x.y, (lane & 16) + c);
            if (r < w && (FWD ? r > c : r < c)) x = cfma(cneg(A[(int64_t)r * ld + c]), xc, x);
        }
        if (r < w && j < nrhs) B[r * ldb + j] = x;
    }
    __syncwarp();
}

// B[rows r0..r1) -= A[rows][c0..c0+w) X (X: w rows, staged in xs), all threads
__device__ __forceinline__ void lu_update_rows(const cplx* A, int ld, int c0, int w, const cplx* xs, int nrhs, cplx* B, int ldb,
                                               int r0, int r1) {
    for (int q = threadIdx.x; q < (r1 - r0) * nrhs; q += blockDim.x) {
        const int r = r0 + q / nrhs, j = q % nrhs;
        cplx x = B[(int64_t)r * ldb + j];
        for (int c = 0; c < w; ++c) x = cfma(cneg(A[(int64_t)r * ld + c0 + c]), xs[c * nrhs + j], x);
        B[(int64_t)r * ldb + j] = x;
    }
}

// Forward (FWD, unit lower) or backward (upper) substitution of B in blocks of NG_LU_TRI rows: a warp solves
// the triangle (staged in shared memory), all threads subtract its columns from the other rows.
// xs: NG_LU_TRI * nrhs values.
template <bool FWD>
__device__ void lu_substitute(const cplx* A, int ld, int N, cplx* B, int ldb, int nrhs, cplx* xs) {
    __shared__ cplx tri_s[NG_LU_TRI * NG_LU_TRI];
    const int nblk = (N + NG_LU_TRI - 1) / NG_LU_TRI;
    for (int q = 0; q < nblk; ++q) {
        const int c0 = (FWD ? q : nblk - 1 - q) * NG_LU_TRI, w = min(NG_LU_TRI, N - c0);
        for (int i = threadIdx.x; i < w * w; i += blockDim.x)
            tri_s[(i / w) * NG_LU_TRI + i % w] = A[(int64_t)(c0 + i / w) * ld + c0 + i % w];
        __syncthreads();
        if (threadIdx.x < 32) lu_tri_block<FWD>(tri_s, NG_LU_TRI, w, B + (int64_t)c0 * ldb, ldb, nrhs, threadIdx.x);
        __syncthreads();
        for (int i = threadIdx.x; i < w * nrhs; i += blockDim.x) xs[i] = B[(int64_t)(c0 + i / nrhs) * ldb + i % nrhs];
        __syncthreads();
        if (FWD) lu_update_rows(A, ld, c0, w, xs, nrhs, B, ldb, c0 + w, N);
        else lu_update_rows(A, ld, c0, w, xs, nrhs, B, ldb, 0, c0);
        __syncthreads();
    }
}

// LU with partial pivoting of the augmented matrix [A | B] (N x (N + nrhs)) and back substitution; one
// block per problem; writes the solution into column block N..N+nrhs.  Panels of PB columns are
// factorised in shared memory; the rest of the matrix is then read and written once per panel, PB
// multiply-adds per element with a lane per column (bound by the FP64 pipe; column by column it was bound
// by the trips to L2: 128 systems of 201 unknowns 8.9 -> 4.1 ms; a refinement solve, 0.73 -> 0.23 ms).
// Shared memory: panel N x PB, NG_LU_TRI * nrhs values, a reduction value and index per warp.
template <int PB>
__global__ void __launch_bounds__(NG_LU_THREADS) k_lu_solve(int N, int nrhs, cplx* ws_A, int* piv, int* status) {
    dep_wait();
    const int ld = N + nrhs;
    cplx* A = ws_A + (int64_t)blockIdx.x * N * ld;
    int* pv = piv + (int64_t)blockIdx.x * N;
    extern __shared__ unsigned char smem_raw[];
    cplx* P = reinterpret_cast<cplx*>(smem_raw);   // [row][PB]
    cplx* xs = P + (size_t)N * PB;
    __shared__ long long rv[NG_LU_THREADS / 32];
    __shared__ int ri[NG_LU_THREADS / 32], prow[PB];
    const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, warp = t >> 5, nw = nt >> 5;
    for (int c0 = 0; c0 < N; c0 += PB) {
        const int w = min(PB, N - c0);
        for (int i = t; i < (N - c0) * PB; i += nt) {
            const int r = c0 + i / PB, c = i % PB;
            P[(size_t)r * PB + c] = c < w ? A[(int64_t)r * ld + c0 + c] : cz();
        }
        __syncthreads();
        for (int c = 0; c < w; ++c) {
            // pivot: the first row of largest magnitude; the diagonal row when none compares (a column of NaN)
            long long best = -1;
            int bi = c0 + c;
            for (int r = c0 + c + t; r < N; r += nt) {
                const long long v = pivot_key(P[(size_t)r * PB + c]);
                if (v > best) { best = v; bi = r; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const long long bo = __shfl_xor_sync(0xffffffffu, best, o);
                const int po = __shfl_xor_sync(0xffffffffu, bi, o);
                if (bo > best || (bo == best && po < bi)) { best = bo; bi = po; }
            }
            if (lane == 0) { rv[warp] = best; ri[warp] = bi; }
            __syncthreads();
            best = rv[0];
            bi = ri[0];
            for (int q = 1; q < nw; ++q)
                if (rv[q] > best || (rv[q] == best && ri[q] < bi)) { best = rv[q]; bi = ri[q]; }
            if (t == 0) {
                if (best <= 0) atomicOr(status, NGF_SINGULAR);
                pv[c0 + c] = prow[c] = bi;
            }
            if (bi != c0 + c && t < PB) {
                const cplx x = P[(size_t)(c0 + c) * PB + t];
                P[(size_t)(c0 + c) * PB + t] = P[(size_t)bi * PB + t];
                P[(size_t)bi * PB + t] = x;
            }
            __syncthreads();
            const cplx inv = cinv(P[(size_t)(c0 + c) * PB + c]);
            for (int r = c0 + c + 1 + t; r < N; r += nt) {
                const cplx f = cmul(P[(size_t)r * PB + c], inv);
                P[(size_t)r * PB + c] = f;
                for (int j = c + 1; j < w; ++j)
                    P[(size_t)r * PB + j] = cfma(cneg(f), P[(size_t)(c0 + c) * PB + j], P[(size_t)r * PB + j]);
            }
            __syncthreads();
        }
        for (int i = t; i < (N - c0) * PB; i += nt) {
            const int r = c0 + i / PB, c = i % PB;
            if (c < w) A[(int64_t)r * ld + c0 + c] = P[(size_t)r * PB + c];
        }
        // the other columns: row interchanges, and right of the panel the rows of U
        for (int j = t; j < ld; j += nt) {
            if (j >= c0 && j < c0 + w) continue;
            for (int c = 0; c < w; ++c) {
                const int p = prow[c];
                if (p == c0 + c) continue;
                const cplx x = A[(int64_t)(c0 + c) * ld + j];
                A[(int64_t)(c0 + c) * ld + j] = A[(int64_t)p * ld + j];
                A[(int64_t)p * ld + j] = x;
            }
            if (j < c0) continue;
            cplx u[PB];
#pragma unroll
            for (int c = 0; c < PB; ++c) {
                if (c >= w) break;
                u[c] = A[(int64_t)(c0 + c) * ld + j];
#pragma unroll
                for (int q = 0; q < c; ++q) u[c] = cfma(cneg(P[(size_t)(c0 + c) * PB + q]), u[q], u[c]);
                A[(int64_t)(c0 + c) * ld + j] = u[c];
            }
        }
        __syncthreads();
        // trailing update: a warp takes 32 columns and every other row chunk of them
        const int ncols = ld - c0 - w, tiles = (ncols + 31) / 32, rows = N - c0 - w;
        const int chunks = max(1, (nw + tiles - 1) / max(1, tiles)), clen = (rows + chunks - 1) / chunks;
        for (int q = warp; q < tiles * chunks; q += nw) {
            const int j = c0 + w + (q % tiles) * 32 + lane;
            if (j >= ld) continue;
            cplx u[PB];
#pragma unroll
            for (int c = 0; c < PB; ++c) u[c] = c < w ? A[(int64_t)(c0 + c) * ld + j] : cz();
            const int r0 = c0 + w + (q / tiles) * clen, r1 = min(N, r0 + clen);
#pragma unroll 2
            for (int r = r0; r < r1; ++r) {
                cplx x = A[(int64_t)r * ld + j];
#pragma unroll
                for (int c = 0; c < PB; ++c) x = cfma(cneg(P[(size_t)r * PB + c]), u[c], x);
                A[(int64_t)r * ld + j] = x;
            }
        }
        __syncthreads();
    }
    lu_substitute<false>(A, ld, N, A + N, ld, nrhs, xs);
}

// The same factorisation for a few larger systems: per column the pivot search, row interchange and multipliers in one
// block per problem (blockIdx.x), then the rank-1 update of the trailing rows and columns over the GPU (problem
// blockIdx.y), at the end the back substitution.  It needs a third of the arithmetic of the inverse.
__global__ void __launch_bounds__(NG_LU_THREADS) k_lu_col(int N, int nrhs, cplx* ws_A, int* piv, int c, int* status) {
    dep_wait();
    const int ld = N + nrhs, t = threadIdx.x, nt = blockDim.x;
    cplx* A = ws_A + (int64_t)blockIdx.x * N * ld;
    __shared__ long long rv[NG_LU_THREADS / 32];
    __shared__ int ri[NG_LU_THREADS / 32];
    long long best = -1;
    int p = c;
    for (int r = c + t; r < N; r += nt) {
        const long long v = pivot_key(A[(int64_t)r * ld + c]);
        if (v > best) { best = v; p = r; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long bo = __shfl_xor_sync(0xffffffffu, best, o);
        const int po = __shfl_xor_sync(0xffffffffu, p, o);
        if (bo > best || (bo == best && po < p)) { best = bo; p = po; }
    }
    if ((t & 31) == 0) { rv[t >> 5] = best; ri[t >> 5] = p; }
    __syncthreads();
    best = rv[0];
    p = ri[0];
    for (int q = 1; q < nt / 32; ++q)
        if (rv[q] > best || (rv[q] == best && ri[q] < p)) { best = rv[q]; p = ri[q]; }
    if (t == 0) {
        if (best <= 0) atomicOr(status, NGF_SINGULAR);
        piv[(int64_t)blockIdx.x * N + c] = p;
    }
    if (p != c)
        for (int j = t; j < ld; j += nt) {
            const cplx x = A[(int64_t)p * ld + j];
            A[(int64_t)p * ld + j] = A[(int64_t)c * ld + j];
            A[(int64_t)c * ld + j] = x;
        }
    __syncthreads();
    const cplx inv = cinv(A[(int64_t)c * ld + c]);
    for (int r = c + 1 + t; r < N; r += nt) A[(int64_t)r * ld + c] = cmul(A[(int64_t)r * ld + c], inv);
}
__global__ void k_lu_rank1(int N, int nrhs, cplx* ws_A, int c) {
    dep_wait();
    const int ld = N + nrhs, w = ld - c - 1;
    cplx* A = ws_A + (int64_t)blockIdx.y * N * ld;
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (int64_t)(N - c - 1) * w) return;
    const int r = c + 1 + (int)(q / w), j = c + 1 + (int)(q % w);
    A[(int64_t)r * ld + j] = cfma(cneg(A[(int64_t)r * ld + c]), A[(int64_t)c * ld + j], A[(int64_t)r * ld + j]);
}
__global__ void __launch_bounds__(NG_LU_THREADS) k_lu_backsub(int N, int nrhs, cplx* ws_A) {
    dep_wait();
    const int ld = N + nrhs;
    cplx* A = ws_A + (int64_t)blockIdx.x * N * ld;
    __shared__ cplx xs[NG_LU_TRI * 8];
    lu_substitute<false>(A, ld, N, A + N, ld, nrhs, xs);
}

// A few problems: the inverse of A by Gauss-Jordan elimination with partial pivoting, one launch per
// column over the whole GPU (a few microseconds each: one pass over an L2-resident matrix), from one
// buffer to the other so that the row interchange needs no second pass.  Each launch also finds the
// next column's pivot: key = magnitude's leading 48 bits (none for a NaN), then the smallest row.  With the inverse, a
// solve is a product (k_gj_apply) instead of 2 N dependent steps of one block: for 402 unknowns and 2
// right-hand sides 1775 -> 9 us, a factorisation with its solve 9.4 -> 2.9 ms.
__device__ __forceinline__ unsigned long long gj_key(cplx x, int r) {
    const long long v = pivot_key(x);
    return ((unsigned long long)(v < 0 ? 0 : v) & ~0xffffull) | (unsigned)(0xffff - r);
}
__global__ void k_gj_first(int N, int ld, const cplx* ws_A, unsigned long long* keys, int* perm) {
    dep_wait();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= N) return;
    perm[(int64_t)blockIdx.y * N + r] = r;
    atomicMax(&keys[(int64_t)blockIdx.y * (N + 1)], gj_key(ws_A[((int64_t)blockIdx.y * N + r) * ld], r));
}
#define NG_GJ_ROWS 8
__global__ void __launch_bounds__(128) k_gj_step(int N, int ld, const cplx* src_, cplx* dst_, int c, unsigned long long* keys,
                                                 int* perm, int* status) {
    dep_wait();
    const int pb = blockIdx.z, j = blockIdx.x * 32 + (threadIdx.x & 31);
    const int r0 = (blockIdx.y * 4 + (threadIdx.x >> 5)) * NG_GJ_ROWS;
    const cplx* src = src_ + (int64_t)pb * N * ld;
    cplx* dst = dst_ + (int64_t)pb * N * ld;
    const unsigned long long key = keys[(int64_t)pb * (N + 1) + c];
    const int p = 0xffff - (int)(key & 0xffff);
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        if (pivot_key(src[(int64_t)p * ld + c]) <= 0) atomicOr(status, NGF_SINGULAR);
        int* pm = perm + (int64_t)pb * N;
        const int x = pm[c];
        pm[c] = pm[p];
        pm[p] = x;
    }
    if (j >= N || r0 >= N) return;
    const cplx inv = cinv(src[(int64_t)p * ld + c]);
    const cplx pr = j == c ? inv : cmul(src[(int64_t)p * ld + j], inv);
    unsigned long long best = 0;
#pragma unroll
    for (int i = 0; i < NG_GJ_ROWS; ++i) {
        const int r = r0 + i;
        if (r >= N) break;
        cplx x;
        if (r == c) x = pr;
        else {
            const int sr = r == p ? c : r;
            x = cfma(cneg(src[(int64_t)sr * ld + c]), pr, j == c ? cz() : src[(int64_t)sr * ld + j]);
            if (j == c + 1 && r > c) best = max(best, gj_key(x, r));
        }
        dst[(int64_t)r * ld + j] = x;
    }
    if (j == c + 1 && best) atomicMax(&keys[(int64_t)pb * (N + 1) + c + 1], best);
}

// ----------------------------------------------------------------------------------------
// Iterative refinement of the Matsubara solve with stored LU factors (from an earlier
// operator): residual r = g + [K * G]^M - G of the current operator (matrix-free, Eqs. cm1/cm2),
// x = (LU)^-1 r with the stored row interchanges, G += x.  The fixed point is the root of the
// current discretised equation; only the convergence path differs from a fresh LU.
// ----------------------------------------------------------------------------------------
// residual of item (m, kb) from the convolution [K * G]^M(m): element (a, b) of r
__device__ __forceinline__ cplx mat_resid_el(cplx gg, cplx kg, cplx gm) { return csub(cadd(gg, kg), gm); }
template <int D>
__global__ void k_mat_resid(Grid g, const cplx* ws_g, const cplx* ws_K, HermV G, cplx* ws_r) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= (int64_t)(g.ntau + 1) * g.nb) return;
    const int kb = (int)(item % g.nb), m = (int)(item / g.nb);
    const int T1 = g.ntau + 1;
    Mat<D> kg = cmat_ws_comp<D>(W, g, ws_K + (int64_t)kb * T1 * D * D, G.mat, m, kb);
    const cplx* gg = ws_g + ((int64_t)kb * T1 + m) * D * D;
    Mat<D> Gm = gmat<D>(G, m, kb);
    cplx* r = ws_r + (int64_t)kb * T1 * D * D;   // row-major [(m a)][b] per problem
    for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b) r[(m * D + a) * D + b] = mat_resid_el(gg[a * D + b], kg.v[a][b], Gm.v[a][b]);
}

// k_mat_resid and k_mat_K with one warp per item: for a few problems the thread form's items are long
// serial sums on a few SMs (one problem, ntau = 200, nf = 2: 331 -> 20 us)
template <int D>
__global__ void __launch_bounds__(128) k_mat_resid_w(Grid g, const cplx* ws_g, const cplx* ws_K, HermV G, cplx* ws_r) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int64_t item = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (item >= (int64_t)(g.ntau + 1) * g.nb) return;
    const int kb = (int)(item % g.nb), m = (int)(item / g.nb), T1 = g.ntau + 1, lane = threadIdx.x & 31;
    const Mat<D> kg = warp_sum_all<D>(cmat_ws_comp_part<D>(W, g, ws_K + (int64_t)kb * T1 * D * D, G.mat, m, kb, lane));
    const int64_t o = ((int64_t)kb * T1 + m) * D * D;
    const Mat<D> Gm = gmat<D>(G, m, kb);
    if (lane == 0)
        for (int a = 0; a < D; ++a)
            for (int b = 0; b < D; ++b) ws_r[o + a * D + b] = mat_resid_el(ws_g[o + a * D + b], kg.v[a][b], Gm.v[a][b]);
}
template <int D>
__global__ void __launch_bounds__(128) k_mat_K_w(Grid g, HermV S, const cplx* ws_g, cplx* ws_K) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int64_t item = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (item >= (int64_t)(g.ntau + 1) * g.nb) return;
    const int kb = (int)(item % g.nb), m = (int)(item / g.nb), T1 = g.ntau + 1, lane = threadIdx.x & 31;
    const Mat<D> K = warp_sum_all<D>(cmat_ws_comp_part<D>(W, g, ws_g + (int64_t)kb * T1 * D * D, S.mat, m, kb, lane));
    if (lane == 0)
        for (int a = 0; a < D; ++a)
            for (int b = 0; b < D; ++b) ws_K[((int64_t)kb * T1 + m) * D * D + a * D + b] = K.v[a][b];
}

// G^M += x: element (m, a, b) <-> x[(m nrhs + a)][b] with N = (ntau+1) nrhs rows
__device__ __forceinline__ int64_t mat_offset(const Comp& mat, int nrhs, int row, int b, int kb) {
    return ((int64_t)(row / nrhs) * nrhs * nrhs + (row % nrhs) * nrhs + b) * mat.ldk + (mat.ldk == 1 ? 0 : kb);
}

// one block per problem: x = U^-1 L^-1 P r in place (r has nrhs columns), then G^M += x and
// *dsum += sum |x|
__global__ void __launch_bounds__(NG_LU_THREADS) k_lu_resolve(Grid g, int N, int nrhs, const cplx* ws_A, const int* piv,
                                                              cplx* ws_r, HermV G, double* dsum) {
    dep_wait();
    const int ld = N + nrhs;
    const cplx* A = ws_A + (int64_t)blockIdx.x * N * ld;
    const int* p = piv + (int64_t)blockIdx.x * N;
    cplx* r = ws_r + (int64_t)blockIdx.x * N * nrhs;
    const int t = threadIdx.x, nt = blockDim.x;
    __shared__ cplx xs[NG_LU_TRI * 8], rs[NG_LU_STAGE];
    __shared__ int ps[NG_LU_STAGE];
    const bool staged = N * nrhs <= NG_LU_STAGE;   // right-hand sides and interchanges fit shared memory
    if (staged) {
        for (int i = t; i < N * nrhs; i += nt) rs[i] = r[i];
        for (int i = t; i < N; i += nt) ps[i] = p[i];
    }
    __syncthreads();
    cplx* x_ = staged ? rs : r;
    const int* p_ = staged ? ps : p;
    if (t < nrhs)   // row interchanges in factorisation order
        for (int c = 0; c < N; ++c) {
            const int q = p_[c];
            if (q != c) { cplx x = x_[c * nrhs + t]; x_[c * nrhs + t] = x_[q * nrhs + t]; x_[q * nrhs + t] = x; }
        }
    __syncthreads();
    lu_substitute<true>(A, ld, N, x_, nrhs, nrhs, xs);
    lu_substitute<false>(A, ld, N, x_, nrhs, nrhs, xs);
    double s = 0.0;
    for (int64_t q = t; q < (int64_t)N * nrhs; q += nt) {
        const int64_t off = mat_offset(G.mat, nrhs, (int)(q / nrhs), (int)(q % nrhs), blockIdx.x);
        const cplx x = x_[q];
        G.mat.p[off] = cadd(G.mat.p[off], x);
        s += sqrt(cabs2(x));
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((t & 31) == 0 && s != 0.0) atomicAdd(dsum, s);
}

// x = A^-1 r with the inverse of k_gj_step (columns in the order of its row interchanges), one warp per
// (row, right-hand side, problem); G^M = x (ADD = false) or G^M += x and *dsum += sum |x|
template <bool ADD>
__global__ void __launch_bounds__(128) k_gj_apply(int N, int ld, int nrhs, const cplx* inv_, const int* perm, const cplx* ws_r, HermV G,
                                                  double* dsum, int* status) {
    dep_wait();
    const int64_t item = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (item >= (int64_t)N * nrhs) return;
    const int pb = blockIdx.y, lane = threadIdx.x & 31, row = (int)(item / nrhs), b = (int)(item % nrhs);
    const cplx* M = inv_ + ((int64_t)pb * N + row) * ld;
    const int* pm = perm + (int64_t)pb * N;
    const cplx* r = ws_r + (int64_t)pb * N * nrhs;
    cplx x = cz();
    for (int j = lane; j < N; j += 32) x = cfma(M[j], r[pm[j] * nrhs + b], x);
    for (int o = 16; o > 0; o >>= 1) {
        x.x += __shfl_xor_sync(0xffffffffu, x.x, o);
        x.y += __shfl_xor_sync(0xffffffffu, x.y, o);
    }
    if (lane != 0) return;
    const int64_t off = mat_offset(G.mat, nrhs, row, b, pb);
    if (ADD) {
        G.mat.p[off] = cadd(G.mat.p[off], x);
        const double s = sqrt(cabs2(x));
        if (s != 0.0) atomicAdd(dsum, s);
    } else {
        G.mat.p[off] = x;
        if (!cfinite(x)) atomicOr(status, NGF_NONFINITE);
    }
}

template <int D>
__global__ void k_mat_store(Grid g, const cplx* ws_A, HermV G, int* status) {
    dep_wait();
    const int T = g.ntau, N = (T + 1) * D, ld = N + D;
    const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= (int64_t)(T + 1) * g.nb) return;
    const int kb = (int)(item % g.nb), m = (int)(item / g.nb);
    const cplx* A = ws_A + (int64_t)kb * N * ld;
    Mat<D> x;
    for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b) x.v[a][b] = A[(int64_t)(m * D + a) * ld + N + b];
    if (!mfinite<D>(x)) atomicOr(status, NGF_NONFINITE);
    st<D>(G.mat, m, kb, x);
}

// ----------------------------------------------------------------------------------------
// start-up (Sec. "Start")
// ----------------------------------------------------------------------------------------
// Retarded columns m = 0..k (one thread per problem) and the common VIDE start-up matrix
// M_{n,l} = D_{n,l}/h + delta_{nl} i(eps_n - mu) + h s_{n,l} i Sigma~^R(n,l) (Eq. vdiff_start):
// the workspace receives inv(M[1..k][1..k]) (kD x kD) and the blocks M[n][0].
template <int D>
__global__ void k_start_ret(Grid g, HermV G, HermV S, FuncV eps, cplx* ws_st, int* status) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int kb = blockIdx.x * blockDim.x + threadIdx.x;
    if (kb >= g.nb) return;
    const int k = W.k, N = k * D;
    cplx A[(NG_KMAX * D) * (NG_KMAX * D)];
    cplx B[(NG_KMAX * D) * (NG_KMAX * D)];
    const Mat<D> mi = meye<D>(make_double2(0.0, -1.0));
    for (int m = 0; m <= k; ++m) {
        Mat<D> y[NG_KMAX + 1];
        for (int l = 0; l < m; ++l) y[l] = mscal<D>(-1.0, mdag<D>(gret<D>(G, m, l, kb)));
        y[m] = mi;
        if (m < k) {
            const int nu = (k - m) * D;
            for (int n = m + 1; n <= k; ++n) {
                Mat<D> e = ldf<D>(eps, n, kb);
                for (int a = 0; a < D; ++a) e.v[a][a].x -= g.mu;
                Mat<D> rhs = mzero<D>();
                for (int l = 0; l <= k; ++l) {
                    // M_{n,l} = i D_{n,l}/h - delta_{nl}(eps_n - mu) - h I_{m,n;l} Sigma~^R(n,l)
                    Mat<D> M = meye<D>(make_double2(0.0, W.D[n][l] / g.h));
                    M = msub<D>(M, mscal<D>(g.h * W.I[m][n][l], gretx<D>(S, n, l, kb)));
                    if (l == n) M = msub<D>(M, e);
                    if (l <= m) rhs = msub<D>(rhs, mmul<D>(M, y[l]));
                    else
                        for (int a = 0; a < D; ++a)
                            for (int b = 0; b < D; ++b) A[((n - m - 1) * D + a) * nu + (l - m - 1) * D + b] = M.v[a][b];
                }
                for (int a = 0; a < D; ++a)
                    for (int c = 0; c < D; ++c) B[((n - m - 1) * D + a) * D + c] = rhs.v[a][c];
            }
            if (dense_solve(A, nu, B, D)) atomicOr(status, NGF_SINGULAR);
            for (int n = m + 1; n <= k; ++n)
                for (int a = 0; a < D; ++a)
                    for (int c = 0; c < D; ++c) y[n].v[a][c] = B[((n - m - 1) * D + a) * D + c];
        }
        for (int n = m; n <= k; ++n) st<D>(G.ret, tri(n) + m, kb, y[n]);
    }
    // VIDE start-up matrix: inverse of M[1..k][1..k] by solving with the identity
    for (int n = 1; n <= k; ++n) {
        Mat<D> e = ldf<D>(eps, n, kb);
        for (int a = 0; a < D; ++a) e.v[a][a].x -= g.mu;
        for (int l = 0; l <= k; ++l) {
            Mat<D> M = meye<D>(cr(W.D[n][l] / g.h));
            M = madd<D>(M, mscal<D>(g.h * W.greg[n][l], mmuli<D>(gretx<D>(S, n, l, kb))));
            if (l == n) M = madd<D>(M, mmuli<D>(e));
            cplx* dst0 = ws_st + (int64_t)kb * (N * N + k * D * D);
            if (l == 0) {
                for (int a = 0; a < D; ++a)
                    for (int b = 0; b < D; ++b) dst0[N * N + (n - 1) * D * D + a * D + b] = M.v[a][b];
            } else {
                for (int a = 0; a < D; ++a)
                    for (int b = 0; b < D; ++b) A[((n - 1) * D + a) * N + (l - 1) * D + b] = M.v[a][b];
            }
        }
    }
    for (int i = 0; i < N; ++i)
        for (int j = 0; j < N; ++j) B[i * N + j] = cr(i == j ? 1.0 : 0.0);
    if (dense_solve(A, N, B, N)) atomicOr(status, NGF_SINGULAR);
    cplx* dst = ws_st + (int64_t)kb * (N * N + k * D * D);
    for (int i = 0; i < N * N; ++i) dst[i] = B[i];
}

// apply the start-up inverse: y_n (n=1..k) = sum_l Minv[n][l] (q_l - M[l][0] y0)
template <int D>
__device__ void start_apply(const cplx* st_ws, int k, const Mat<D>* q, const Mat<D>& y0, Mat<D>* y) {
    const int N = k * D;
    Mat<D> rhs[NG_KMAX];
    for (int l = 0; l < k; ++l) {
        Mat<D> M0;
        for (int a = 0; a < D; ++a)
            for (int b = 0; b < D; ++b) M0.v[a][b] = st_ws[N * N + l * D * D + a * D + b];
        rhs[l] = msub<D>(q[l], mmul<D>(M0, y0));
    }
    for (int n = 0; n < k; ++n) {
        Mat<D> acc = mzero<D>();
        for (int l = 0; l < k; ++l) {
            Mat<D> Mi;
            for (int a = 0; a < D; ++a)
                for (int b = 0; b < D; ++b) Mi.v[a][b] = st_ws[(n * D + a) * N + l * D + b];
            mfma<D>(acc, Mi, rhs[l]);
        }
        y[n] = acc;
    }
}

template <int D>
__global__ void k_start_tv(Grid g, HermV G, HermV S, const cplx* ws_st, int* status) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= (int64_t)(g.ntau + 1) * g.nb) return;
    const int kb = (int)(item % g.nb), m = (int)(item / g.nb);
    const int k = W.k, N = k * D;
    Mat<D> y0 = mcscal<D>(make_double2(0.0, (double)g.sig), gmat<D>(G, g.ntau - m, kb));  // i xi G^M(beta - tau_m)
    Mat<D> q[NG_KMAX], y[NG_KMAX];
    for (int n = 1; n <= k; ++n) q[n - 1] = q_tv<D>(W, g, G, S, n, m, kb);
    start_apply<D>(ws_st + (int64_t)kb * (N * N + k * D * D), k, q, y0, y);
    st<D>(G.tv, m, kb, y0);
    for (int n = 1; n <= k; ++n) {
        if (!mfinite<D>(y[n - 1])) atomicOr(status, NGF_NONFINITE);
        st<D>(G.tv, (int64_t)n * (g.ntau + 1) + m, kb, y[n - 1]);
    }
}

template <int D>
__global__ void k_start_les(Grid g, HermV G, HermV S, const cplx* ws_st, int* status) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int k = W.k, N = k * D;
    const int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= (int64_t)(k + 1) * g.nb) return;
    const int kb = (int)(item % g.nb), n = (int)(item / g.nb);
    Mat<D> y0 = mscal<D>(-1.0, mdag<D>(gtv<D>(G, g, n, 0, kb)));
    Mat<D> q[NG_KMAX], y[NG_KMAX];
    for (int m = 1; m <= k; ++m) q[m - 1] = q_lesA_part<D>(W, g, G, S, m, n, kb, 0, 1);
    start_apply<D>(ws_st + (int64_t)kb * (N * N + k * D * D), k, q, y0, y);
    st<D>(G.les, tri(n) + 0, kb, y0);
    for (int m = 1; m <= n; ++m) {
        if (!mfinite<D>(y[m - 1])) atomicOr(status, NGF_NONFINITE);
        st<D>(G.les, tri(n) + m, kb, y[m - 1]);
    }
}

// ----------------------------------------------------------------------------------------
// The start-up kernels with one warp per item (nf <= 4): a few problems leave the thread forms to a few
// lanes with serial sums over tau and dense solves of (k nf)^2 (one problem, nf = 2, ntau = 200: 4.04 -> 0.28 ms
// for the three).  Same formulas; sums over the lanes.
// ----------------------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ Mat<D> start_matrix_el(const NgWeights& W, const Grid& g, const HermV& S, const FuncV& eps, int n, int l,
                                                  int kb) {   // M_{n,l} of Eq. vdiff_start
    Mat<D> M = meye<D>(cr(W.D[n][l] / g.h));
    M = madd<D>(M, mscal<D>(g.h * W.greg[n][l], mmuli<D>(gretx<D>(S, n, l, kb))));
    if (l == n) {
        Mat<D> e = ldf<D>(eps, n, kb);
        for (int a = 0; a < D; ++a) e.v[a][a].x -= g.mu;
        M = madd<D>(M, mmuli<D>(e));
    }
    return M;
}

template <int D>
__global__ void __launch_bounds__(32) k_start_ret_w(Grid g, HermV G, HermV S, FuncV eps, cplx* ws_st, int* status) {
    dep_wait();
    constexpr int NM = NG_KMAX * D;
    const NgWeights& W = c_W[g.k - 1];
    const int kb = blockIdx.x, lane = threadIdx.x, k = W.k, N = k * D;
    __shared__ cplx A[NM * NM], B[NM * NM], f[NM], y[NG_KMAX + 1][D][D];
    for (int m = 0; m <= k; ++m) {
        if (lane == 0) {
            for (int l = 0; l < m; ++l) {
                const Mat<D> x = mscal<D>(-1.0, mdag<D>(gret<D>(G, m, l, kb)));
                for (int a = 0; a < D; ++a)
                    for (int b = 0; b < D; ++b) y[l][a][b] = x.v[a][b];
            }
            for (int a = 0; a < D; ++a)
                for (int b = 0; b < D; ++b) y[m][a][b] = make_double2(0.0, a == b ? -1.0 : 0.0);
        }
        __syncwarp();
        if (m < k) {
            const int nu = (k - m) * D;
            // lane -> block (n, l): l > m into A; l <= m: -M_{n,l} y_l, added up by the lane of (n, 0) below
            for (int q = lane; q < (k - m) * (k - m); q += 32) {
                const int n = m + 1 + q / (k - m), l = m + 1 + q % (k - m);
                Mat<D> M = meye<D>(make_double2(0.0, W.D[n][l] / g.h));
                M = msub<D>(M, mscal<D>(g.h * W.I[m][n][l], gretx<D>(S, n, l, kb)));
                if (l == n) {
                    Mat<D> e = ldf<D>(eps, n, kb);
                    for (int a = 0; a < D; ++a) e.v[a][a].x -= g.mu;
                    M = msub<D>(M, e);
                }
                for (int a = 0; a < D; ++a)
                    for (int b = 0; b < D; ++b) A[((n - m - 1) * D + a) * nu + (l - m - 1) * D + b] = M.v[a][b];
            }
            for (int n = m + 1 + lane; n <= k; n += 32) {
                Mat<D> rhs = mzero<D>();
                for (int l = 0; l <= m; ++l) {
                    Mat<D> M = meye<D>(make_double2(0.0, W.D[n][l] / g.h)), yl;
                    M = msub<D>(M, mscal<D>(g.h * W.I[m][n][l], gretx<D>(S, n, l, kb)));
                    for (int a = 0; a < D; ++a)
                        for (int b = 0; b < D; ++b) yl.v[a][b] = y[l][a][b];
                    rhs = msub<D>(rhs, mmul<D>(M, yl));
                }
                for (int a = 0; a < D; ++a)
                    for (int c = 0; c < D; ++c) B[((n - m - 1) * D + a) * D + c] = rhs.v[a][c];
            }
            __syncwarp();
            if (warp_dense_solve(A, nu, B, D, f, lane) && lane == 0) atomicOr(status, NGF_SINGULAR);
            __syncwarp();
        }
        for (int n = m + lane; n <= k; n += 32) {
            Mat<D> x;
            for (int a = 0; a < D; ++a)
                for (int c = 0; c < D; ++c) x.v[a][c] = n == m ? y[m][a][c] : B[((n - m - 1) * D + a) * D + c];
            st<D>(G.ret, tri(n) + m, kb, x);
        }
        __syncwarp();   // the next column reads G^R(m + 1, .) back
    }
    // VIDE start-up matrix: inverse of M[1..k][1..k], and the blocks M[n][0]
    cplx* dst = ws_st + (int64_t)kb * (N * N + k * D * D);
    for (int q = lane; q < k * (k + 1); q += 32) {
        const int n = 1 + q / (k + 1), l = q % (k + 1);
        const Mat<D> M = start_matrix_el<D>(W, g, S, eps, n, l, kb);
        for (int a = 0; a < D; ++a)
            for (int b = 0; b < D; ++b)
                (l == 0 ? dst[N * N + (n - 1) * D * D + a * D + b] : A[((n - 1) * D + a) * N + (l - 1) * D + b]) = M.v[a][b];
    }
    for (int i = lane; i < N * N; i += 32) B[i] = cr(i / N == i % N ? 1.0 : 0.0);
    __syncwarp();
    if (warp_dense_solve(A, N, B, N, f, lane) && lane == 0) atomicOr(status, NGF_SINGULAR);
    __syncwarp();
    for (int i = lane; i < N * N; i += 32) dst[i] = B[i];
}

// y_n = sum_l Minv[n][l] (q_l - M[l][0] y0), one element (n, a, b) per lane and turn; q: the warp's scratch
// with the sources, overwritten
template <int D>
__device__ __forceinline__ void start_apply_w(const cplx* st_ws, int k, cplx (*q)[D][D], const Mat<D>& y0, int lane,
                                              const Comp& out, int64_t (*elem)(const Grid&, int, int), const Grid& g, int col, int nlast,
                                              int kb, int* status) {
    const int N = k * D;
    cplx(*y0s)[D] = q[NG_KMAX];
    if (lane == 0)
        for (int a = 0; a < D; ++a)
            for (int b = 0; b < D; ++b) y0s[a][b] = y0.v[a][b];
    __syncwarp();
    for (int i = lane; i < k * D * D; i += 32) {
        const int l = i / (D * D), a = i / D % D, b = i % D;
        cplx x = q[l][a][b];
        for (int c = 0; c < D; ++c) x = cfma(cneg(st_ws[N * N + l * D * D + a * D + c]), y0s[c][b], x);
        q[l][a][b] = x;
    }
    __syncwarp();
    for (int i = lane; i < nlast * D * D; i += 32) {
        const int n = i / (D * D), a = i / D % D, b = i % D;
        cplx x = cz();
        for (int l = 0; l < k; ++l)
            for (int c = 0; c < D; ++c) x = cfma(st_ws[(n * D + a) * N + l * D + c], q[l][c][b], x);
        if (!cfinite(x)) atomicOr(status, NGF_NONFINITE);
        cel(out, elem(g, n + 1, col), a, b, D, kb) = x;
    }
}
__device__ inline int64_t start_el_tv(const Grid& g, int n, int m) { return (int64_t)n * (g.ntau + 1) + m; }
__device__ inline int64_t start_el_les(const Grid&, int m, int n) { return tri(n) + m; }

template <int D>
__global__ void __launch_bounds__(128) k_start_tv_w(Grid g, HermV G, HermV S, const cplx* ws_st, int* status) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int64_t item = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (item >= (int64_t)(g.ntau + 1) * g.nb) return;
    const int kb = (int)(item % g.nb), m = (int)(item / g.nb), k = W.k, N = k * D, lane = threadIdx.x & 31;
    __shared__ cplx sh[4][NG_KMAX + 1][D][D];
    cplx(*q)[D][D] = sh[threadIdx.x >> 5];
    const Mat<D> y0 = mcscal<D>(make_double2(0.0, (double)g.sig), gmat<D>(G, g.ntau - m, kb));  // i xi G^M(beta - tau_m)
    for (int n = 1; n <= k; ++n) {
        const Mat<D> x = warp_sum_all<D>(q_tv_part<D>(W, g, G, S, n, m, kb, lane));
        if (lane == 0)
            for (int a = 0; a < D; ++a)
                for (int b = 0; b < D; ++b) q[n - 1][a][b] = x.v[a][b];
    }
    __syncwarp();
    if (lane == 0) st<D>(G.tv, m, kb, y0);
    start_apply_w<D>(ws_st + (int64_t)kb * (N * N + k * D * D), k, q, y0, lane, G.tv, start_el_tv, g, m, k, kb, status);
}

template <int D>
__global__ void __launch_bounds__(128) k_start_les_w(Grid g, HermV G, HermV S, const cplx* ws_st, int* status) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int k = W.k, N = k * D, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int kb = blockIdx.x % g.nb, n = blockIdx.x / g.nb;   // one block: a warp per source row in turn
    __shared__ cplx q[NG_KMAX + 1][D][D];
    const Mat<D> y0 = mscal<D>(-1.0, mdag<D>(gtv<D>(G, g, n, 0, kb)));
    for (int m = 1 + warp; m <= k; m += 4) {
        const Mat<D> x = warp_sum_all<D>(q_lesA_part<D>(W, g, G, S, m, n, kb, lane, 32));
        if (lane == 0)
            for (int a = 0; a < D; ++a)
                for (int b = 0; b < D; ++b) q[m - 1][a][b] = x.v[a][b];
    }
    __syncthreads();
    if (warp != 0) return;
    if (lane == 0) st<D>(G.les, tri(n) + 0, kb, y0);
    start_apply_w<D>(ws_st + (int64_t)kb * (N * N + k * D * D), k, q, y0, lane, G.les, start_el_les, g, n, n, kb, status);
}
