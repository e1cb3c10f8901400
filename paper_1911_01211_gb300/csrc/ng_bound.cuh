// Boundary of a time step for batches of one-orbital problems (nf = 1, n > 2k): the (A) rows
// m = n-k..n of the lesser column with one lane per problem.
//
// k_step_boundary takes a block per problem, reads the problem-innermost store with a stride of a
// whole batch between lanes and runs 2(k+1) block reductions one after the other; its time was
// latency and half-used sectors.  Here a warp's lanes are 32 neighbouring problems: each value of
// row n and of the column is loaded once, in whole lines, and enters all k+1 rows' sums.  Those are
// bound by the FP64 pipe (18 multiply-adds per index and problem; an FP64 warp instruction takes 64
// clocks of its quarter SM, so the sums are spread over all of them and the serial rest is kept short); a shared self-energy's weighted
// values come from shared memory.  512 problems, n = 240, ntau = 800: 133 -> 77 us;
// 64 problems, n = 40, ntau = 100: 62 -> 22 us (the retarded start-up runs beside the bulk items).
#pragma once

#include "ng_stepsplit.cuh"

#define NG_B1_ROWS (NG_KMAX + 1)
#define NG_B1_SEG 32            // indices staged at a time

// weighted self-energy values of row m at index j: source over the real times, over tau, history
// (l < m0).  q = -i h C^<_2 - i (C^<_3): the factors of q_lesA_part are folded in.
__device__ __forceinline__ void bnd1_values(const NgWeights& W, const Grid& g, const HermV& S, int n, int m, int j, int kb,
                                            cplx& c2, cplx& c3, cplx& hs) {
    const int T = g.ntau, m0 = n - W.k;
    c2 = c3 = hs = cz();
    if (j <= n) {
        const cplx x = cscal(g.h * gw(W, n, j), gles<1>(S, m, j, kb).v[0][0]);
        c2 = make_double2(x.y, -x.x);
    }
    if (j <= T) c3 = cscal((double)g.sig * g.htau * gw(W, T, j), gtv<1>(S, g, m, j, kb).v[0][0]);
    if (j < m0) hs = cscal(gw(W, m, j), gret<1>(S, m, j, kb).v[0][0]);
}

// block (32 problems, chunk of indices): part[((chunk * 2 NR) + i) nb + kb], i = r: source of row r,
// NR + r: its partial history
template <bool SHARED>
static __global__ void __launch_bounds__(128) k_bnd1_sums(Grid g, int n, HermV G, HermV S, int len, cplx* part) {
    dep_wait();
    constexpr int NR = NG_B1_ROWS;
    const NgWeights& W = c_W[g.k - 1];
    const int k = W.k, T = g.ntau, m0 = n - k, J = max(n, T) + 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int kb = blockIdx.x * 32 + lane, kc = min(kb, g.nb - 1);
    __shared__ cplx sm[4 * 2 * NR * 32];   // staged values [index][3][row]; then the warps' sums
    cplx q[NR], h[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) q[r] = h[r] = cz();
    const int jend = min(J, ((int)blockIdx.y + 1) * len);
    for (int js = blockIdx.y * len; js < jend; js += NG_B1_SEG) {
        if (SHARED) {
            __syncthreads();
            for (int i = threadIdx.x; i < NG_B1_SEG * NR; i += 128) {
                const int j = js + i / NR, r = i % NR;
                cplx c2 = cz(), c3 = cz(), hs = cz();
                if (r <= k && j < jend) bnd1_values(W, g, S, n, m0 + r, j, 0, c2, c3, hs);
                cplx* o = sm + (i / NR) * 3 * NR + r;
                o[0] = c2; o[NR] = c3; o[2 * NR] = hs;
            }
            __syncthreads();
        }
        const int je = min(js + NG_B1_SEG, jend);
        for (int j = js + warp; j < je; j += 4) {
            cplx gr = cz(), gt = cz(), gl = cz();
            if (j <= n) gr = cconj(G.ret.p[(tri(n) + j) * G.ret.ldk + kc]);
            if (j <= T) gt = cconj(G.tv.p[((int64_t)n * (T + 1) + T - j) * G.tv.ldk + kc]);
            if (j < m0)   // G^<(0, n) = -conj G^tv(n, 0) is stored by k_bnd1_fin
                gl = j == 0 ? les0_of_tv<1>(g, G, n, kc).v[0][0] : G.les.p[(tri(n) + j) * G.les.ldk + kc];
            const cplx* o = sm + (j - js) * 3 * NR;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                if (r > k) break;
                cplx c2, c3, hs;
                if (SHARED) { c2 = o[r]; c3 = o[NR + r]; hs = o[2 * NR + r]; }
                else bnd1_values(W, g, S, n, m0 + r, j, kc, c2, c3, hs);
                if (j <= n) q[r] = cfma(c2, gr, q[r]);
                if (j <= T) q[r] = cfma(c3, gt, q[r]);
                if (j < m0) h[r] = cfma(hs, gl, h[r]);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        sm[((warp * 2 + 0) * NR + r) * 32 + lane] = q[r];
        sm[((warp * 2 + 1) * NR + r) * 32 + lane] = h[r];
    }
    __syncthreads();
    if (kb >= g.nb) return;
    for (int i = warp; i < 2 * NR; i += 4) {
        cplx v = sm[i * 32 + lane];
        for (int w = 1; w < 4; ++w) v = cadd(v, sm[(w * 2 * NR + i) * 32 + lane]);
        part[((int64_t)blockIdx.y * 2 * NR + i) * g.nb + kb] = v;
    }
}

// G^<(0, n), the chunk partials in chunk order, then the k+1 serial (A) steps of a problem in one lane:
//   y_r = M_r^-1 (b_r - sum_{d<r} c_rd y_d),  c_rd = a_{r-d}/h + i h w Sigma^R(m_r, m_d),
// with everything but the recurrence itself (15 multiply-adds and 6 products) spread over the warps.
#define NG_B1_WARPS 12
static __global__ void __launch_bounds__(32 * NG_B1_WARPS) k_bnd1_fin(Grid g, int n, HermV G, HermV S, FuncV eps, int nchunk,
                                                                      const cplx* part, int* status) {
    dep_wait();
    constexpr int NR = NG_B1_ROWS;
    static_assert(NG_B1_WARPS == 2 * NR, "a warp per partial sum");
    const NgWeights& W = c_W[g.k - 1];
    const int k = W.k, m0 = n - k;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int kb = blockIdx.x * 32 + lane, kc = min(kb, g.nb - 1);
    const double hinv = 1.0 / g.h;
    __shared__ cplx qh[2 * NR][32], Mi[NR][32], cf[NR * NR][32], base[NR][32];
    auto col = [&](int l) { return G.les.p[(tri(n) + l) * G.les.ldk + kc]; };   // l = m0-k..m0-1: from the bulk
    {
        cplx v = cz();
        for (int c = 0; c < nchunk; ++c) v = cadd(v, part[((int64_t)c * 2 * NR + warp) * g.nb + kc]);
        qh[warp][lane] = v;
    }
    cplx bd = cz();
    if (warp < NR && warp <= k) {   // BDF terms of row m0 + warp that lie below m0
        for (int l = warp + 1; l <= k; ++l) bd = make_double2(fma(W.a[l], col(m0 + warp - l).x, bd.x), fma(W.a[l], col(m0 + warp - l).y, bd.y));
    } else if (warp >= NR && warp - NR <= k) {
        const int r = warp - NR;
        int sing = 0;
        Mi[r][lane] = minv<1>(step_matrix<1>(W, g, S, eps, m0 + r, kc), &sing).v[0][0];
        if (sing) atomicOr(status, NGF_SINGULAR);
        for (int d = 0; d < r; ++d) {
            const cplx x = cscal(g.h * gw(W, m0 + r, m0 + d), gret<1>(S, m0 + r, m0 + d, kc).v[0][0]);
            cf[r * NR + d][lane] = make_double2(fma(W.a[r - d], hinv, -x.y), x.x);
        }
    }
    __syncthreads();
    if (warp < NR && warp <= k) {
        const cplx q = qh[warp][lane], h = qh[NR + warp][lane];   // q - bd / h - i h hist
        base[warp][lane] = make_double2(fma(g.h, h.y, fma(-hinv, bd.x, q.x)), fma(-g.h, h.x, fma(-hinv, bd.y, q.y)));
    }
    __syncthreads();
    if (warp != 0 || kb >= g.nb) return;
    G.les.p[tri(n) * G.les.ldk + kb] = les0_of_tv<1>(g, G, n, kb).v[0][0];
    cplx y[NR];
    bool ok = true;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        if (r > k) break;
        cplx acc = base[r][lane];
#pragma unroll
        for (int d = 0; d < r; ++d) acc = cfma(cneg(cf[r * NR + d][lane]), y[d], acc);
        y[r] = cmul(Mi[r][lane], acc);
        ok = ok && cfinite(y[r]);
        G.les.p[(tri(n) + m0 + r) * G.les.ldk + kb] = y[r];
    }
    if (!ok) atomicOr(status, NGF_NONFINITE);
}
