// History sums of the uneven batch by digit products (ng_histu.cu): the row vectors of a step and the
// closing of its bulk items.
#pragma once

#include "ng_hist.cuh"
#include "ng_histu.h"
#include "ng_ubatch.cuh"

// ---- row vectors ----------------------------------------------------------------------------------
__device__ __forceinline__ cplx histu_vec_value(const NgWeights& W, const UProb& p, int n, int vec, int o, int i) {
    const int D = p.g.nf, k = W.k, T = p.g.ntau, j = i / D, c = i % D;
    if (vec == 4) {
        if (j > T) return cz();
        const cplx x = uel(p.S.tv, (int64_t)n * (T + 1) + j, D, o, c, 0);
        return j <= k ? cscal(W.omega[j], x) : (j >= T - k ? cscal(W.omega[T - j], x) : x);
    }
    if (vec == 3) return j > T ? cz() : cscal(gw(W, T, j), uel(p.S.tv, (int64_t)n * (T + 1) + T - j, D, o, c, 0));
    if (j >= n) return cz();
    if (vec == 2) {
        const cplx x = uel(p.S.les, tri(n) + j, D, c, o, 0);
        return j <= k ? cscal(W.omega[j], x) : x;
    }
    const cplx x = uel(p.S.ret, tri(n) + j, D, o, c, 0);
    if (vec == 1 || vec == 5) return cscal(gw(W, n, j), x);
    return j >= n - k ? cscal(W.omega[n - j], x) : x;
}

// block (128 elements, problem, 8 vector + output): values, scales and digits.  Each chunk of the contraction (the kt
// tiles of a task) has the scale of its largest element, which every block of 128 elements finds by itself; it
// touches two chunks at most (16 tiles and more each).  Blocks of vector NGU_NVEC write Y.
static __global__ void __launch_bounds__(128) k_histu_vec(const __grid_constant__ HistUTab tab) {
    dep_wait();
    const UProb& p = tab.src[tab.prob[blockIdx.y]];
    const int D = p.g.nf, vec = blockIdx.z >> 3, o = blockIdx.z & 7, n = tab.n, tid = threadIdx.x;
    const int len = (vec == 3 || vec == 4 ? p.g.ntau + 1 : n) * D;
    if (vec == NGU_NVEC) {
        HistUGeo q;
        histu_geo(D, p.g.ntau, n, q);
        cplx* y = (cplx*)(tab.base + tab.off[blockIdx.y] + q.conv);
        const int T = p.g.ntau, DD = D * D;
        for (int i = (o * gridDim.x + blockIdx.x) * 128 + tid; i < (2 * T + 1) * DD; i += 8 * gridDim.x * 128) {
            const int d = i / DD - T, ab = i % DD;   // Y(0) is not used
            const cplx x = p.G.mat.p[(int64_t)(d > 0 ? T - d : -d) * DD + ab];
            y[i] = d > 0 ? cscal((double)p.g.sig, x) : x;
        }
        return;
    }
    if (o >= D || (int)blockIdx.x * 128 >= (len + 127) / 128 * 128) return;
    const NgWeights& W = c_W[p.g.k - 1];
    __shared__ int smax[2];
    __shared__ __align__(16) __half dig[8][2][8][4][2][2][2];   // as NGH_DIG_B
    HistUGeo q;
    histu_geo(D, p.g.ntau, n, q);
    char* base = tab.base + tab.off[blockIdx.y];
    if (tid == 0) {
        smax[0] = smax[1] = 0;
        if (blockIdx.x + blockIdx.y + blockIdx.z == 0) *tab.next = 0;
        if (blockIdx.x == 0 && blockIdx.z == 0)
            tab.probs[blockIdx.y] = HistUProb{p.G, p.S, p.g, p.minv, (cplx*)base, (uint4*)(base + q.tab), (int*)(base + q.vexp),
                                              (cplx*)(base + q.conv), (cplx*)(base + q.part), q};
    }
    __syncthreads();
    const int ke = histu_vec_kt(q, vec) * 16, ch0 = (int)blockIdx.x * 128 / ke, ch1 = ((int)blockIdx.x * 128 + 127) / ke;
    for (int ch = ch0; ch <= ch1; ++ch) {
        int e = 0;
#pragma unroll 4
        for (int i = ch * ke + tid; i < min(len, (ch + 1) * ke); i += 128) {
            const cplx x = histu_vec_value(W, p, n, vec, o, i);
            e = max(e, max(__double2hiint(x.x) >> 20 & 2047, __double2hiint(x.y) >> 20 & 2047));
        }
        atomicMax(&smax[ch - ch0], e);
    }
    __syncthreads();
    if (tid <= ch1 - ch0 && (ch0 + tid) * ke < len)   // each block of a chunk writes the same value
        ((int*)(base + q.vexp))[(vec * D + o) * q.vch + ch0 + tid] = smax[tid] == 2047 ? -1 : max(smax[tid], 128);
    const int i0 = blockIdx.x * 128 + tid, F = max(smax[i0 / ke - ch0], 128);
    const cplx x = i0 < len ? histu_vec_value(W, p, n, vec, o, i0) : cz();
    ((cplx*)base)[((int64_t)vec * D + o) * q.lenp + i0] = x;
    hist_digits(x, F, histu_conj(vec), tid & 15, dig[tid >> 4]);
    __syncthreads();
    uint4* dst = (uint4*)(base + q.tab) + (((int64_t)vec * D + o) * (q.lenp / 16) + blockIdx.x * 8) * 64;
    for (int i = tid; i < 8 * 64; i += 128) dst[i] = ((const uint4*)&dig[0][0][0][0][0][0][0])[i];
}

// ---- closing -----------------------------------------------------------------------------------------
// sum of the chunks of a set at free index (time i, orbital r), output o
__device__ __forceinline__ cplx histu_sum(const HistUProb& p, int set, int i, int r, int o) {
    const int D = p.g.nf;
    const cplx* q = p.part + p.q.poff[set] + ((int64_t)i * D + r) * D + o;
    cplx x = cz();
    for (int c = 0; c < p.q.chunks[set]; ++c) x = cadd(x, q[(int64_t)c * p.q.free_[set] * D]);
    return x;
}

// u_qtv with the long parts of both convolutions from the units
template <int D>
__device__ __forceinline__ cplx u_qtv_hist(const NgWeights& W, const HistUProb& p, int n, int m, int a, int b) {
    const Grid& g = p.g;
    const int k = W.k, T = g.ntau;
    const int64_t row = (int64_t)n * (T + 1);
    cplx c[2];   // over [0, m], over [m, T]: e steps from the end of the axis, where index 0 is
#pragma unroll
    for (int z = 0; z < 2; ++z) {
        const int e = z ? T - m : m;
        cplx x = cz();
        auto add = [&](double w, int js, int jg) {
#pragma unroll
            for (int q = 0; q < D; ++q)
                x = cfma(cscal(w, uel(p.S.tv, row + (z ? T - js : js), D, a, q, 0)), uel(p.G.mat, z ? jg : T - jg, D, q, b, 0), x);
        };
        if (e <= k) {
            for (int j = 0; j <= k; ++j)
                for (int l = 0; l <= k; ++l) add(W.R[e][j][l], l, j);
        } else if (e <= 2 * k + 1) {
            for (int l = 0; l <= e; ++l) add(W.greg[e][l], e - l, l);
        } else {
            for (int l = 0; l <= k; ++l) add(W.omega[l], e - l, l);
        }
        c[z] = x;
    }
    return cscal(g.htau, cmulmi(cadd(cadd(cscal((double)g.sig, c[0]), c[1]), histu_sum(p, 6, m, b, a))));
}

// right-hand side of element (a, b) of a bulk item, as u_rhs, with the history sums from the units
template <int D>
__device__ cplx u_rhs_hist(const NgWeights& W, const HistUProb& p, int n, int task, int m, int a, int b) {
    const Grid& g = p.g;
    const HermV &G = p.G, &S = p.S;
    const int k = W.k, T1 = g.ntau + 1;
    if (task == 2) {
        const int L = n - m;
        if (L <= 2 * k + 1) return u_rhs<D>(W, g, G, S, n, task, m, a, b, 0);
        cplx acc = histu_sum(p, 0, m, b, a), bdf = cz();
        for (int l = 0; l <= k; ++l)
#pragma unroll
            for (int c = 0; c < D; ++c)
                acc = cfma(cscal(W.omega[l], uel(S.ret, tri(n) + m + l, D, a, c, 0)), uel(G.ret, tri(m + l) + m, D, c, b, 0), acc);
        for (int l = 1; l <= k; ++l) bdf = cadd(bdf, cscal(W.a[l], uel(G.ret, tri(n - l) + m, D, a, b, 0)));
        return csub(cscal(-1.0 / g.h, bdf), cscal(g.h, cmuli(acc)));
    }
    if (task == 1) {
        cplx bdf = cz();
        for (int l = 1; l <= k; ++l) bdf = cadd(bdf, cscal(W.a[l], uel(G.tv, (int64_t)(n - l) * T1 + m, D, a, b, 0)));
        cplx r = u_qtv_hist<D>(W, p, n, m, a, b);
        r = csub(r, cscal(1.0 / g.h, bdf));
        return csub(r, cscal(g.h, cmuli(histu_sum(p, 4, m, b, a))));
    }
    cplx c1 = cz();
    if (m <= 2 * k + 1) {
        for (int j = 0; j <= max(m, k); ++j)
#pragma unroll
            for (int c = 0; c < D; ++c)
                c1 = cfma(cscal(W.greg[m][j], uretx(G, m, j, D, a, c, 0)), uel(S.les, tri(n) + j, D, c, b, 0), c1);
    } else {
        c1 = histu_sum(p, 1, m, a, b);
        for (int j = m - k; j <= m; ++j)
#pragma unroll
            for (int c = 0; c < D; ++c)
                c1 = cfma(cscal(W.omega[m - j], uel(G.ret, tri(m) + j, D, a, c, 0)), uel(S.les, tri(n) + j, D, c, b, 0), c1);
    }
    const cplx c3 = histu_sum(p, 5, m, a, b);
    cplx hist = csub(histu_sum(p, 2, m, a, b), cconj(histu_sum(p, 3, m, a, b)));
#pragma unroll
    for (int c = 0; c < D; ++c)   // l = m
        hist = cfma(uel(G.les, tri(m) + m, D, a, c, 0), cconj(p.vec[((int64_t)D + b) * p.q.lenp + m * D + c]), hist);
    cplx bdf = cz();
    for (int l = 1; l <= k; ++l) bdf = cadd(bdf, cscal(W.a[l], uel(G.les, tri(n - l) + m, D, a, b, 0)));
    const cplx q = csub(cscal(g.h, cmuli(c1)), cscal((double)g.sig * g.htau, c3));
    return cadd(csub(q, cscal(1.0 / g.h, bdf)), cscal(g.h, cmuli(hist)));
}

// k_ubulk with the sums from the tasks: what is left is the quadrature's ends, the BDF terms and the product with
// M_n^-1 (16 clusters of 1..8 orbitals, n = 500, ntau = 300: 0.19 ms)
template <int D>
__device__ __forceinline__ void u_close_block(const HistUProb& P, int n, int lblk, int nles, int ntv, int* status) {
    const NgWeights& W = c_W[P.g.k - 1];
    constexpr int DD = D * D;
    const int ipb = blockDim.x / DD;  // items per block
    int task, base;
    if (lblk < nles) { task = 0; base = lblk; }
    else if (lblk < nles + ntv) { task = 1; base = lblk - nles; }
    else { task = 2; base = lblk - nles - ntv; }
    const int t = threadIdx.x;
    const int li = t / DD, ab = t % DD, a = ab / D, b = ab % D;
    const int col = base * ipb + li, k = W.k;
    const int ncol = task == 0 ? n - k - 1 : (task == 1 ? P.g.ntau + 1 : n - k), m = task == 0 ? col + 1 : col;
    const bool valid = (li < ipb) && (col < ncol);
    extern __shared__ cplx rhs[];   // blockDim.x entries
    if (t < ipb * DD) rhs[t] = valid ? u_rhs_hist<D>(W, P, n, task, m, a, b) : cz();
    __syncthreads();
    if (!valid) return;
    const cplx* rr = rhs + li * DD;
    cplx y = cz();
#pragma unroll
    for (int c = 0; c < D; ++c)   // y = rhs (M_n^-1)^dagger (lesser), M_n^-1 rhs
        y = task == 0 ? cfma(rr[a * D + c], cconj(P.minv[b * D + c]), y) : cfma(P.minv[a * D + c], rr[c * D + b], y);
    if (!cfinite(y)) atomicOr(status, NGF_NONFINITE);
    const Comp& dst = task == 0 ? P.G.les : (task == 1 ? P.G.tv : P.G.ret);
    ust(dst, task == 1 ? (int64_t)n * (P.g.ntau + 1) + m : tri(n) + m, D, a, b, 0, y);
}
static __global__ void __launch_bounds__(256) k_histu_close(const HistUProb* probs, UTable tab, int* status) {
    dep_wait();
    int i = 0;
    while (i + 1 < tab.np && (int)blockIdx.x >= tab.start[i + 1]) ++i;
    const HistUProb& P = probs[i];
    const int lblk = blockIdx.x - tab.start[i];
    switch (P.g.nf) {
        case 1: u_close_block<1>(P, tab.n, lblk, tab.nles[i], tab.ntv[i], status); break;
        case 2: u_close_block<2>(P, tab.n, lblk, tab.nles[i], tab.ntv[i], status); break;
        case 4: u_close_block<4>(P, tab.n, lblk, tab.nles[i], tab.ntv[i], status); break;
        default: u_close_block<8>(P, tab.n, lblk, tab.nles[i], tab.ntv[i], status); break;
    }
}
