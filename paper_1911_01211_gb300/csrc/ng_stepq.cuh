// Time step for middling batches of one-orbital problems: P = 4 or 8 lanes per bulk item.
//
// FP64 is issued per warp and quarter SM, one instruction in 64 clocks on this part, so what a small step
// costs is its number of FP64 warp instructions: a warp per item (k_step_bulk_w) spends 10 additions per
// sum on adding its lanes and a closing step per item, a thread per item (k_step_bulk) fills too few
// quarter SMs.  Here a warp holds 32 / P neighbouring problems of one column (whole sectors of the
// problem-innermost store); the P lanes of an item take every P-th term of all its sums, which with the
// BDF terms and their factors go into one accumulator, added by log2 P butterflies.  64 problems, n = 40,
// ntau = 100: 66 -> 30 us, the whole step 97 -> 62 us.
#pragma once

#include "ng_stepsplit.cuh"

// f(l, w_{L,l}) for every P-th term l = 0..lmax of a Gregory row L, from p on
template <int P, class F>
__device__ __forceinline__ void greg_for_part(const NgWeights& W, int L, int lmax, int p, F&& f) {
    const int k = W.k;
    if (L <= 2 * k + 1) {
        for (int l = p; l <= lmax; l += P) f(l, W.greg[L][l]);
        return;
    }
    for (int l = p; l <= k; l += P) f(l, W.omega[l]);
    for (int l = L - k + p; l <= lmax; l += P) f(l, W.omega[L - l]);
#pragma unroll 4
    for (int l = k + 1 + p; l <= L - k - 1; l += P) f(l, 1.0);
}

// this part's terms of -i (C^tv_2 + C^tv_3)[S, 1, G^M](n, tau_m), as q_tv
template <int P>
__device__ __forceinline__ cplx q_tv_lanes(const NgWeights& W, const Grid& g, const HermV& G, const HermV& S, int n, int m, int kb,
                                           int p) {
    const int k = W.k, T = g.ntau, kk = (k + 1) * (k + 1);
    auto s = [&](int j) { return gtv<1>(S, g, n, j, kb).v[0][0]; };
    auto gm = [&](int j) { return gmat<1>(G, j, kb).v[0][0]; };
    cplx c2 = cz(), c3 = cz();
    if (m <= k) {
        for (int i = p; i < kk; i += P) c2 = cfma(cscal(W.R[m][i / (k + 1)][i % (k + 1)], s(i % (k + 1))), gm(T - i / (k + 1)), c2);
    } else {
        greg_for_part<P>(W, m, m, p, [&](int l, double w) { c2 = cfma(cscal(w, s(m - l)), gm(T - l), c2); });
    }
    if (m >= T - k) {
        for (int i = p; i < kk; i += P) c3 = cfma(cscal(W.R[T - m][i / (k + 1)][i % (k + 1)], s(T - i % (k + 1))), gm(i / (k + 1)), c3);
    } else {
        greg_for_part<P>(W, T - m, T - m, p, [&](int l, double w) { c3 = cfma(cscal(w, s(m + l)), gm(l), c3); });
    }
    const cplx v = cadd(cscal((double)g.sig, c2), c3);
    return make_double2(g.htau * v.y, -g.htau * v.x);
}

// Items (column, problem) as in k_step_bulk; warp = (column, group of 32 / P problems).  The first w_pre
// warps run the boundary's retarded start-up of a problem each.  tvq: the FFT pre-pass, or NULL: the direct
// sums of the left-mixing source.
template <int P>
static __global__ void __launch_bounds__(128) k_step_bulk_q(Grid g, int n, HermV G, HermV S, FuncV eps, const cplx* minv_ws,
                                                            int w_pre, int c_les, int c_tv, int c_ret, const cplx* tvq, int* status) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    constexpr int Q = 32 / P;
    const int k = W.k, T = g.ntau, lane = threadIdx.x & 31, q = lane % Q, p = lane / Q;
    int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w < w_pre) {
        __shared__ cplx sh[4][bnd_pre_scratch<1>()];
        bnd_pre_warp<1>(W, g, n, G, S, eps, (int)w, sh[threadIdx.x >> 5], lane, status);
        return;
    }
    w -= w_pre;
    const int ngrp = (g.nb + Q - 1) / Q;
    int col = (int)(w / ngrp), task;
    const int kb = min((int)(w % ngrp) * Q + q, g.nb - 1);   // lanes past the batch repeat its last problem
    const bool own = (int)(w % ngrp) * Q + q < g.nb;
    if (col < c_les) task = 0;
    else if ((col -= c_les) < c_tv) task = 1;
    else if ((col -= c_tv) < c_ret) task = 2;
    else return;
    const int m = task == 0 ? col + 1 : col;
    const Comp& X = task == 0 ? G.les : (task == 1 ? G.tv : G.ret);
    auto at = [&](int i) { return task == 1 ? (int64_t)i * (T + 1) + m : tri(i) + m; };
    cplx acc = cz(), rhs = cz();   // acc: sums that enter with a factor h i (lesser) or -h i
    if (task == 0) {
        const cplx* sl = S.les.p + tri(n) * S.les.ldk;
        auto les = [&](int j) { return sl[(int64_t)j * S.les.ldk + (S.les.ldk == 1 ? 0 : kb)]; };
        if (m <= k) {
            for (int j = p; j <= k; j += P) acc = cfma(cscal(W.greg[m][j], gretx<1>(G, m, j, kb).v[0][0]), les(j), acc);
        } else {
            greg_for_part<P>(W, m, m, p, [&](int j, double x) { acc = cfma(cscal(x, gret<1>(G, m, j, kb).v[0][0]), les(j), acc); });
        }
        greg_for_part<P>(W, n, n - 1, p, [&](int l, double x) {
            const cplx gl = l >= m ? G.les.p[(tri(l) + m) * G.les.ldk + kb] : cneg(cconj(G.les.p[(tri(m) + l) * G.les.ldk + kb]));
            acc = cfma(cscal(x, gl), cconj(gret<1>(S, n, l, kb).v[0][0]), acc);
        });
        cplx c3 = cz();
        greg_for_part<P>(W, T, T, p, [&](int j, double x) {
            c3 = cfma(cscal(x, gtv<1>(G, g, m, j, kb).v[0][0]), cconj(gtv<1>(S, g, n, T - j, kb).v[0][0]), c3);
        });
        rhs = cadd(cscal(g.h, cmuli(acc)), cscal(-(double)g.sig * g.htau, c3));
    } else if (task == 1) {
        greg_for_part<P>(W, n, n - 1, p, [&](int j, double x) {
            acc = cfma(cscal(x, gret<1>(S, n, j, kb).v[0][0]), gtv<1>(G, g, j, m, kb).v[0][0], acc);
        });
        rhs = cscal(g.h, cmulmi(acc));
        if (!tvq) rhs = cadd(rhs, q_tv_lanes<P>(W, g, G, S, n, m, kb, p));
        else if (p == 0) rhs = cadd(rhs, q_tv_fft<1>(W, g, G, S, n, m, kb, tvq).v[0][0]);
    } else {
        const int L = n - m;
        greg_for_part<P>(W, L, L - 1, p, [&](int l, double x) {
            acc = cfma(cscal(x, gret<1>(S, n, m + l, kb).v[0][0]), gret<1>(G, m + l, m, kb).v[0][0], acc);
        });
        rhs = cscal(g.h, cmulmi(acc));
    }
    const double hinv = -1.0 / g.h;
    for (int l = 1 + p; l <= k; l += P) {
        const cplx x = X.p[at(n - l) * X.ldk + kb];
        const double a = hinv * W.a[l];
        rhs = make_double2(fma(a, x.x, rhs.x), fma(a, x.y, rhs.y));
    }
#pragma unroll
    for (int o = Q; o < 32; o <<= 1) {
        rhs.x += __shfl_xor_sync(0xffffffffu, rhs.x, o);
        rhs.y += __shfl_xor_sync(0xffffffffu, rhs.y, o);
    }
    const cplx Mi = minv_ws[kb], y = cmul(rhs, task == 0 ? cconj(Mi) : Mi);
    if (p != 0 || !own) return;
    if (!cfinite(y)) atomicOr(status, NGF_NONFINITE);
    X.p[at(n) * X.ldk + kb] = y;
}
