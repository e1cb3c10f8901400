// The row vectors of a step for the digit-product history sums (ng_hist.cu) and the sums of each
// item of a step from the units (nf = 1).
//
// With the self-energy slice n (S, and Scc for its lesser column) and W's quadrature weights:
//   vector 0   S^R(n, j), weighted by the end weights of j >= n - k      retarded columns
//   vector 1   w_{n,j} S^R(n, j)                    left-mixing columns, lesser rows and columns
//   vector 2   Scc^<(j, n), weighted by the end weights of j <= k       C^<_1 of row m
//   vector 3   w_{T,j} S^tv(n, T - j)                                   C^<_3 of row m
// The history kernel leaves out the diagonal band of the triangles (retarded: j - m <= k, whose
// terms carry the weights of the other end of the quadrature; lesser: j = m, which belongs to one
// of the two sums only); the closing adds those terms.
#pragma once

#include <cuda_fp16.h>

#include "ng_hist.h"
#include "ng_step.cuh"

struct HistRow {         // slice n of the row functions: element j at p[j * ld + (ld == 1 ? 0 : kb)]
    const cplx *ret, *les, *tv;
    int ld_ret, ld_les, ld_tv;
};

__device__ __forceinline__ cplx hist_vec_value(const NgWeights& W, const HistRow& S, int n, int T, int vec, int j, int kb) {
    const int k = W.k;
    if (vec == 3) {
        if (j > T) return cz();
        return cscal(gw(W, T, j), S.tv[(int64_t)(T - j) * S.ld_tv + (S.ld_tv == 1 ? 0 : kb)]);
    }
    if (j >= n) return cz();
    if (vec == 2) {
        const cplx x = S.les[(int64_t)j * S.ld_les + (S.ld_les == 1 ? 0 : kb)];
        return j <= k ? cscal(W.omega[j], x) : x;
    }
    const cplx x = S.ret[(int64_t)j * S.ld_ret + (S.ld_ret == 1 ? 0 : kb)];
    if (vec == 1) return cscal(gw(W, n, j), x);
    return j >= n - k ? cscal(W.omega[n - j], x) : x;
}

// 64 fraction bits of |x| on the scale 2^(F-1022) of the largest element
__device__ __forceinline__ uint64_t hist_fixed(double x, int F) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 2047), s = F - e;
    if (e == 0 || s > 63) return 0;
    return ((b << 11) | 0x8000000000000000ull) >> s;
}

// Digits of element i (8 half + 2t + {0,1}) of its block of 16 on the scale F (2047: a non-finite vector, zeros),
// balanced: -128..127, the leading one up to 128; layout of NGH_DIG_B
__device__ __forceinline__ void hist_digits(cplx x, int F, bool conj, int i, __half (&dig)[2][8][4][2][2][2]) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const double v = c ? x.y : x.x;
        const bool neg = v < 0.0;
        const uint64_t M = F == 2047 ? 0 : hist_fixed(v, F) >> 1;
        int carry = 0;
#pragma unroll
        for (int d = 7; d >= 0; --d) {
            int b = (int)(M >> (56 - 8 * d) & 255) + carry;
            carry = 0;
            if (b >= 128 && d > 0) { b -= 256; carry = 1; }
            const __half q = __int2half_rn(neg ? -b : b), m = __int2half_rn(neg ? b : -b);
            auto at = [&](int part, int f) -> __half& { return dig[part][d][(i & 7) >> 1][i >> 3][f][i & 1]; };
            if (c == 0) at(0, 0) = at(1, 1) = q;
            else { at(1, 0) = conj ? m : q; at(0, 1) = conj ? q : m; }
        }
    }
}

// FP64 values, scale and digits of the row vectors.  A block takes 128 elements of one vector, with their own
// scale, and of KK problems (KK = 1: vectors shared by all problems).
template <int KK>
static __global__ void __launch_bounds__(256) k_hist_vec(HistWs w, HistRow S) {
    dep_wait();
    const NgWeights& W = c_W[w.k - 1];
    constexpr int PE = KK == 1 ? NGH_BLK : 256 / KK, NP = NGH_BLK / PE;   // elements of a pass, passes
    __shared__ int smax[KK];
    __shared__ __align__(16) __half dig[KK][PE / 16][2][8][4][2][2][2];   // as NGH_DIG_B
    const int vec = blockIdx.z, tid = threadIdx.x, kk = tid % KK, el = tid / KK;
    const int kv = blockIdx.y * KK + kk, kvc = min(kv, w.nv - 1);
    const int len = vec == 3 ? w.T + 1 : w.n, j0 = blockIdx.x * NGH_BLK;
    if (j0 >= len) return;
    if (tid == 0 && blockIdx.x + blockIdx.y + blockIdx.z == 0) *w.next = 0;
    if (tid < KK) smax[tid] = 0;
    __syncthreads();
    cplx x[NP];
    int e = 0;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        x[p] = el < PE ? hist_vec_value(W, S, w.n, w.T, vec, j0 + p * PE + el, kvc) : cz();
        e = max(e, max(__double2hiint(x[p].x) >> 20 & 2047, __double2hiint(x[p].y) >> 20 & 2047));
    }
    atomicMax(&smax[kk], e);
    __syncthreads();
    const int F = max(smax[kk], 128);
    if (el == 0 && kv < w.nv) w.vexp[(vec * w.nv + kv) * (w.lenp / NGH_BLK) + blockIdx.x] = F == 2047 ? -1 : F;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const int j = j0 + p * PE + el;
        if (el < PE) {
            if (kv < w.nv) w.vec[((int64_t)vec * w.nv + kv) * w.lenp + j] = x[p];
            hist_digits(x[p], F, vec == 3, j & 15, dig[kk][el / 16]);   // the left-mixing row vector enters conjugated
        }
        __syncthreads();
        constexpr int NU = KK * (PE / 16) * 64;   // uint4 of the pass
        for (int i = tid; i < NU; i += 256) {
            const int q = i / (PE / 16 * 64), r = i % (PE / 16 * 64), kq = blockIdx.y * KK + q;
            if (kq < w.nv)
                w.tab[(((int64_t)vec * w.nv + kq) * (w.lenp / 16) + (j0 + p * PE) / 16) * 64 + r] =
                    ((const uint4*)&dig[q][0][0][0][0][0][0][0])[r];
        }
        __syncthreads();
    }
}

// column c, row r of a unit's sums
__device__ __forceinline__ cplx hist_col(const HistWs& w, int64_t unit, int c, int kb) {
    return w.part[(unit * NGH_PART + c) * w.nb + kb];
}
__device__ __forceinline__ cplx hist_row(const HistWs& w, int64_t unit, int r, int kb) {
    return w.part[(unit * NGH_PART + NGH_BLK + r) * w.nb + kb];
}

// sum_{j<n} of the retarded column m (n - m > k): unit weights of the interior, Gregory weights at
// both ends
__device__ __forceinline__ cplx hist_ret_sum(const NgWeights& W, const HistWs& w, const HermV& G, const HermV& S, int n,
                                             int m, int kb) {
    const int k = W.k, L = n - m;
    cplx acc = cz();
    if (L <= 2 * k + 1) {
        for (int l = 0; l < L; ++l)
            acc = cfma(cscal(W.greg[L][l], gret<1>(S, n, m + l, kb).v[0][0]), gret<1>(G, m + l, m, kb).v[0][0], acc);
        return acc;
    }
    const int bj = m / NGH_BLK, c = m % NGH_BLK;
    for (int bi = bj; bi < w.nbr; ++bi) acc = cadd(acc, hist_col(w, hist_unit_ret(w, bi, bj), c, kb));
    for (int l = 0; l <= k; ++l)
        acc = cfma(cscal(W.omega[l], gret<1>(S, n, m + l, kb).v[0][0]), gret<1>(G, m + l, m, kb).v[0][0], acc);
    return acc;
}

__device__ __forceinline__ cplx hist_tv_sum(const HistWs& w, int m, int kb) {
    cplx acc = cz();
    const int bj = m / NGH_BLK, c = m % NGH_BLK;
    for (int bi = 0; bi < w.nbr; ++bi) acc = cadd(acc, hist_col(w, hist_unit_tv(w, bi, bj), c, kb));
    return acc;
}

// the three sums of the lesser item m: C^<_1 (without h), C^<_3 (without i xi h_tau) and the history
__device__ __forceinline__ void hist_les_sums(const NgWeights& W, const HistWs& w, const HermV& G, const cplx* sl, int ld_sl,
                                              const cplx* v1, int n, int m, int kb, cplx& c1, cplx& c3, cplx& hist) {
    const int k = W.k, bm = m / NGH_BLK, r = m % NGH_BLK, T1 = w.T + 1;
    auto les = [&](int j) { return sl[(int64_t)j * ld_sl + (ld_sl == 1 ? 0 : kb)]; };
    c1 = c3 = hist = cz();
    if (m <= 2 * k + 1) {
        for (int j = 0; j <= max(m, k); ++j) c1 = cfma(cscal(W.greg[m][j], gretx<1>(G, m, j, kb).v[0][0]), les(j), c1);
    } else {
        for (int bj = 0; bj <= bm; ++bj) c1 = cadd(c1, hist_row(w, hist_unit_ret(w, bm, bj), r, kb));
        for (int j = m - k; j <= m; ++j) c1 = cfma(cscal(W.omega[m - j], gret<1>(G, m, j, kb).v[0][0]), les(j), c1);
    }
    for (int bj = 0; bj * NGH_BLK < T1; ++bj) c3 = cadd(c3, hist_row(w, hist_unit_tv(w, bm, bj), r, kb));
    for (int bi = bm; bi < w.nbr; ++bi) hist = cadd(hist, hist_col(w, hist_unit_les(w, bi, bm), r, kb));
    cplx lo = cz();   // l < m: -conj(sum_l v1(l) G^<(l, m))
    for (int bj = 0; bj <= bm; ++bj) lo = cadd(lo, hist_row(w, hist_unit_les(w, bm, bj), r, kb));
    hist = csub(hist, cconj(lo));
    hist = cfma(G.les.p[(tri(m) + m) * G.les.ldk + kb], cconj(v1[m]), hist);
}
