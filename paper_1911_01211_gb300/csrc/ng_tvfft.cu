// The Toeplitz part of the left-mixing Matsubara source of a time step by FFT.
//
// The source of the left-mixing row at step n is q(m) = -i (C^tv_2 + C^tv_3)[Sigma, 1, G^M](n, m)
// (Eqs. ctv2, ctv3).  Away from the ends of the tau axis (2k+1 < m < ntau - 2k-1) its Gregory weights
// factor into end weights omega of S and of K, so both pieces together are one correlation
//   F(m) = sum_{j=0..ntau} S(j) K(j - m),   S(j) = omega_j' Sigma^tv(t_n, tau_j), j' = min(j, ntau - j),
//   K(d) = omega_{-d} xi G^M(tau_{ntau+d}) (d < 0),  K(0) = omega_0 (xi G^M(beta) + G^M(0)),
//   K(d) = omega_d G^M(tau_d) (d > 0),   omega_j = 1 for j > k,
// which this kernel evaluates for all m at once as a cyclic convolution of length L >= 2 ntau + 1
// (a power of two): forward transforms of S and of the reversed K, their (matrix) product per
// frequency, one inverse transform.  In the 2k+2 columns next to either end the quadrature differs
// from F by O(k) terms (short rows, boundary formulas), which the time-step kernels add (q_tv_fft in
// ng_step.cuh).  (With unit weights here every column needed 4(k+1) correction terms: 144 FP64
// instructions of the closing of each left-mixing item.)  For the F32C kernels the warps here add them (`ends`), a column
// each in turn: with them k_step_bulk32p lost the schedule of its main loops (128 problems, n = 100, ntau = 900: 0.46 ms, 0.31
// without, whole steps 634 / 464 us; 12 problems 551 / 452).  Not for the others: the lanes of a warp per column are not
// as well used as those of a thread per item, and steps of 512 problems, n = 40, ntau = 100 took 175 instead of 149 us.
//
// One block per problem; the transforms are radix-2 decimation in time in shared memory, bit-reversed
// in, natural out; the spectra are multiplied and put back into bit-reversed order in one pass.  They
// are bound by the FP64 pipe, so a butterfly is six fused multiply-adds (v = a - w b, u = 2 a - v)
// and the first two stages have no multiplication: 31 instead of 44 instructions per point at L = 2048.  A
// self-energy shared by the batch is transformed once, by one block ahead (24 us at L = 2048), which pays from
// 64 problems on.  512 problems, ntau = 800: 328 -> 194 us, and k_hist_close 210 -> 88 us.
// Twiddles exp(-2 pi i p / L) come from a table built once per length.
#include "ng_tvfft.h"

namespace {

constexpr int kThreads = 256;
constexpr int kMaxThreads = 768;
// With the ends a warp for each of the 24 columns while every block has an SM to itself (152; 48 registers let an SM hold
// one block of 768 threads or two of 512), else as many blocks as fit
inline int fft_threads(int nb, bool ends) { return !ends || nb > 304 ? kThreads : nb <= 152 ? kMaxThreads : 512; }

__global__ void k_twiddle(cplx* tw, int L) {
    dep_wait();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= L / 2) return;
    double s, c;
    sincospi(-2.0 * (double)p / (double)L, &s, &c);
    tw[p] = make_double2(c, s);
}

// in place, bit-reversed order in, natural out, unscaled; kernel exp(-2 pi i jk / L), conjugate for INV
template <bool INV>
__device__ void fft_dit(cplx* x, const cplx* __restrict__ tw, int L) {
    // stages of span 1 and 2: twiddles 1 and -i (L is at least 16)
    for (int t = threadIdx.x; t < (L >> 2); t += blockDim.x) {
        const cplx a = x[4 * t], b = x[4 * t + 1], c = x[4 * t + 2], d = x[4 * t + 3];
        const cplx s = cadd(a, b), u = csub(a, b), v = cadd(c, d), w = INV ? cmuli(csub(c, d)) : cmulmi(csub(c, d));
        x[4 * t] = cadd(s, v);
        x[4 * t + 1] = cadd(u, w);
        x[4 * t + 2] = csub(s, v);
        x[4 * t + 3] = csub(u, w);
    }
    __syncthreads();
    for (int span = 4; span < L; span <<= 1) {
        const int str = (L >> 1) / span;
        for (int t = threadIdx.x; t < (L >> 1); t += blockDim.x) {
            const int pos = t & (span - 1), i = ((t - pos) << 1) + pos, j = i + span;
            const cplx a = x[i], b = x[j];
            cplx w = __ldg(&tw[pos * str]);
            if (INV) w.y = -w.y;
            const cplx v = make_double2(fma(w.y, b.y, fma(-w.x, b.x, a.x)), fma(-w.y, b.x, fma(-w.x, b.y, a.y)));
            x[j] = v;
            x[i] = make_double2(fma(2.0, a.x, -v.x), fma(2.0, a.y, -v.y));
        }
        __syncthreads();
    }
}

__device__ __forceinline__ cplx el(const Comp& c, int64_t e, int ab, int kb) {
    return c.p[(e * c.dd + ab) * c.ldk + (c.ldk == 1 ? 0 : kb)];
}

// S(i), i = 0..L-1, element e of problem kb
__device__ __forceinline__ cplx s_value(const NgWeights& W, const Grid& g, int64_t rowS, const Comp& Stv, int i, int e, int kb) {
    if (i > g.ntau) return cz();
    const int d = min(i, g.ntau - i);
    const cplx x = el(Stv, rowS + i, e, kb);
    return d <= g.k ? cscal(W.omega[d], x) : x;
}

// spectra of the nf^2 elements of a shared S: FS[e L + frequency]
__global__ void __launch_bounds__(1024) k_tvsrc_s(Grid g, NgWeights W, int n, Comp Stv, const cplx* tw, int L, cplx* FS) {
    dep_wait();
    extern __shared__ cplx sm[];
    const int lg = 31 - __clz(L), e = blockIdx.x;
    for (int i = threadIdx.x; i < L; i += blockDim.x)
        sm[__brev(i) >> (32 - lg)] = s_value(W, g, (int64_t)n * (g.ntau + 1), Stv, i, e, 0);
    __syncthreads();
    fft_dit<false>(sm, tw, L);
    for (int i = threadIdx.x; i < L; i += blockDim.x) FS[(int64_t)e * L + i] = sm[i];
}

// Q[(m nf^2 + a nf + b) nb + kb] = F_ab(m), m = 0..ntau, for problem kb = blockIdx.x; FSg: the spectra of a
// shared S, or NULL; ends: with the corrections of the columns next to the ends
template <int D>
__global__ void __launch_bounds__(kMaxThreads) k_tvsrc_fft(Grid g, NgWeights W, int n, Comp Stv, Comp Gmat, const cplx* tw, int L,
                                                        const cplx* FSg, bool ends, cplx* Q) {
    dep_wait();
    extern __shared__ cplx sm[];
    constexpr int DD = D * D;
    cplx* FK = sm;            // [c b][L]: reversed K_cb, then the product P_ab in place
    cplx* FS = sm + DD * L;   // [a c][L]: S_ac
    const int kb = blockIdx.x, T = g.ntau, lg = 31 - __clz(L);
    const double xi = (double)g.sig;
    const int64_t rowS = (int64_t)n * (T + 1);
    for (int e = 0; e < DD; ++e)
        for (int i = threadIdx.x; i < L; i += blockDim.x) {
            const int r = __brev(i) >> (32 - lg);
            if (!FSg) FS[e * L + r] = s_value(W, g, rowS, Stv, i, e, kb);
            cplx v = cz();
            if (i == 0) v = cadd(cscal(xi, el(Gmat, T, e, kb)), el(Gmat, 0, e, kb));
            else if (i <= T) v = cscal(xi, el(Gmat, T - i, e, kb));          // K(-i)
            else if (i >= L - T) v = el(Gmat, L - i, e, kb);                 // K(L - i)
            const int d = min(i, L - i);
            FK[e * L + r] = d <= g.k ? cscal(W.omega[d], v) : v;
        }
    __syncthreads();
    for (int e = 0; e < DD; ++e) fft_dit<false>(FK + e * L, tw, L);
    if (!FSg)
        for (int e = 0; e < DD; ++e) fft_dit<false>(FS + e * L, tw, L);
    // product per frequency, to the bit-reversed position: frequencies i and rev(i) change places
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        const int r = __brev(i) >> (32 - lg);
        if (r < i) continue;
        cplx p[2][D][D];
#pragma unroll
        for (int z = 0; z < 2; ++z) {
            const int f = z ? r : i;
#pragma unroll
            for (int a = 0; a < D; ++a)
#pragma unroll
                for (int b = 0; b < D; ++b) {
                    cplx q = cz();
#pragma unroll
                    for (int c = 0; c < D; ++c)
                        q = cfma(FSg ? __ldg(&FSg[(a * D + c) * L + f]) : FS[(a * D + c) * L + f], FK[(c * D + b) * L + f], q);
                    p[z][a][b] = q;
                }
        }
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
            for (int b = 0; b < D; ++b) {
                FK[(a * D + b) * L + r] = p[0][a][b];
                FK[(a * D + b) * L + i] = p[1][a][b];
            }
    }
    __syncthreads();
    for (int e = 0; e < DD; ++e) fft_dit<true>(FK + e * L, tw, L);
    const double inv = 1.0 / (double)L;
    const int k = g.k, edge = 2 * k + 2, lane = threadIdx.x & 31;
    for (int e = 0; e < DD; ++e)
        for (int m = threadIdx.x; m <= T; m += blockDim.x)
            if (!ends || min(m, T - m) >= edge) Q[((int64_t)m * DD + e) * g.nb + kb] = cscal(inv, FK[e * L + m]);
    const int ncol = ends ? min(T + 1, 2 * edge) : 0;
    for (int c = threadIdx.x >> 5; c < ncol; c += blockDim.x >> 5) {
        const int m = c < edge ? c : T - (ncol - 1 - c), L3 = T - m;
        auto om = [&](int l) { return l <= k ? W.omega[l] : 1.0; };
        auto ws = [&](int j) { return om(min(j, T - j)); };   // F's weight of S(j)
        cplx x[D][D];
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
            for (int b = 0; b < D; ++b) x[a][b] = cz();
        auto add = [&](double w, int js, int jg) {   // w S(js) G^M(jg)
#pragma unroll
            for (int a = 0; a < D; ++a)
#pragma unroll
                for (int q = 0; q < D; ++q) {
                    const cplx v = cscal(w, el(Stv, rowS + js, a * D + q, kb));
#pragma unroll
                    for (int b = 0; b < D; ++b) x[a][b] = cfma(v, el(Gmat, jg, q * D + b, kb), x[a][b]);
                }
        };
        // C2: sum_l w_{m,l} S(m-l) xi G^M(T-l)
        auto t2 = [&](int l, double w) { add(xi * (w - om(l) * ws(m - l)), m - l, T - l); };
        if (m <= k) {
            for (int i = lane; i < (k + 1) * (k + 1); i += 32) add(xi * W.R[m][i / (k + 1)][i % (k + 1)], i % (k + 1), T - i / (k + 1));
            for (int l = lane; l <= m; l += 32) t2(l, 0.0);
        } else if (m <= 2 * k + 1) {
            for (int l = lane; l <= m; l += 32) t2(l, W.greg[m][l]);
        } else {
            for (int l = lane; l <= m - T + k; l += 32) t2(l, gw(W, m, l));   // the weights of the end j = T
        }
        // C3: sum_l w_{T-m,l} S(m+l) G^M(l)
        auto t3 = [&](int l, double w) { add(w - om(l) * ws(m + l), m + l, l); };
        if (L3 <= k) {
            for (int i = lane; i < (k + 1) * (k + 1); i += 32) add(W.R[L3][i / (k + 1)][i % (k + 1)], T - i % (k + 1), i / (k + 1));
            for (int l = lane; l <= L3; l += 32) t3(l, 0.0);
        } else if (L3 <= 2 * k + 1) {
            for (int l = lane; l <= L3; l += 32) t3(l, W.greg[L3][l]);
        } else {
            for (int l = lane; l <= k - m; l += 32) t3(l, gw(W, L3, l));      // the weights of the end j = 0
        }
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
            for (int b = 0; b < D; ++b) {
                cplx y = x[a][b];
                for (int o = 16; o > 0; o >>= 1) {
                    y.x += __shfl_xor_sync(0xffffffffu, y.x, o);
                    y.y += __shfl_xor_sync(0xffffffffu, y.y, o);
                }
                if (lane == 0) Q[((int64_t)m * DD + a * D + b) * g.nb + kb] = cadd(cscal(inv, FK[(a * D + b) * L + m]), y);
            }
    }
}

template <int D>
cudaError_t launch_d(const Grid& g, const NgWeights& W, int n, const Comp& Stv, const Comp& Gmat, const cplx* tw, cplx* Q,
                     bool ends, cudaStream_t s) {
    const int L = tvfft_length(g.ntau);
    const size_t one = sizeof(cplx) * (size_t)D * D * L;
    const bool shared = tvfft_shared(g, Stv.ldk);
    cplx* FS = shared ? Q + (size_t)(g.ntau + 1) * D * D * g.nb : nullptr;
    cudaError_t e;
    if (shared) {
        const size_t sm = sizeof(cplx) * (size_t)L;
        if ((e = smem_limit(k_tvsrc_s))) return e;
        dep_launch(k_tvsrc_s, D * D, L >= 2048 ? 1024 : L / 2, sm, s)(g, W, n, Stv, tw, L, FS);
        if ((e = cudaGetLastError())) return e;
    }
    const size_t sm = shared ? one : 2 * one;
    if ((e = smem_limit(k_tvsrc_fft<D>))) return e;
    dep_launch(k_tvsrc_fft<D>, g.nb, fft_threads(g.nb, ends), sm, s)(g, W, n, Stv, Gmat, tw, L, FS, ends, Q);
    return cudaGetLastError();
}

}  // namespace

bool tvfft_shared(const Grid& g, int ldk) { return ldk == 1 && g.nb >= 64; }
size_t tvfft_out_bytes(const Grid& g, int ldk) {
    const size_t dd = (size_t)g.nf * g.nf;
    return sizeof(cplx) * dd * ((size_t)(g.ntau + 1) * g.nb + (tvfft_shared(g, ldk) ? tvfft_length(g.ntau) : 0));
}

int tvfft_length(int ntau) {
    int L = 1;
    while (L < 2 * ntau + 1) L <<= 1;
    return L;
}

size_t tvfft_smem_bytes(int nf, int ntau) { return (size_t)2 * nf * nf * tvfft_length(ntau) * sizeof(cplx); }

bool tvfft_supported(int nf, int ntau) {
    return (nf == 1 || nf == 2) && tvfft_smem_bytes(nf, ntau) <= NG_TVFFT_MAX_SMEM;
}

cudaError_t tvfft_twiddles(cplx* tw, int L, cudaStream_t s) {
    dep_launch(k_twiddle, (L / 2 + 255) / 256, 256, 0, s)(tw, L);
    return cudaGetLastError();
}

cudaError_t tvfft_launch(const Grid& g, const NgWeights& W, int n, const Comp& Stv, const Comp& Gmat, const cplx* tw, cplx* Q,
                         bool ends, cudaStream_t s) {
    return g.nf == 1 ? launch_d<1>(g, W, n, Stv, Gmat, tw, Q, ends, s) : launch_d<2>(g, W, n, Stv, Gmat, tw, Q, ends, s);
}
