// Closing of a Dyson time step whose history sums come from the digit products (nf = 1).
#pragma once

#include "ng_hist.cuh"
#include "ng_stepsplit.cuh"

// Items as in k_step_bulk (nf = 1): lesser m = 1..n-k-1, left-mixing m = 0..ntau, retarded
// m = 0..n-k-1; problem fastest.  The first nb_pre blocks run the boundary's retarded start-up, a warp
// per problem: it reads only the self-energy and eps and writes G^R(n, n-k..n), which no item reads.
static __global__ void __launch_bounds__(128) k_hist_close(Grid g, int n, HermV G, HermV S, FuncV eps, HistWs w,
                                                           const cplx* minv_ws, int nb_pre, int nb_les, int nb_tv,
                                                           const cplx* tvq, int* status) {
    dep_wait();
    const NgWeights& W = c_W[g.k - 1];
    const int k = W.k;
    int blk = blockIdx.x, task;
    if (blk < nb_pre) {
        __shared__ cplx sh[4][bnd_pre_scratch<1>()];
        const int warp = threadIdx.x >> 5, kb = blk * 4 + warp;
        if (kb < g.nb) bnd_pre_warp<1>(W, g, n, G, S, eps, kb, sh[warp], threadIdx.x & 31, status);
        return;
    }
    blk -= nb_pre;
    if (blk < nb_les) task = 0;
    else if ((blk -= nb_les) < nb_tv) task = 1;
    else { blk -= nb_tv; task = 2; }
    const int64_t item = (int64_t)blk * blockDim.x + threadIdx.x;
    const int kb = (int)(item % g.nb);
    const int64_t col = item / g.nb;
    const int ncol = task == 0 ? n - k - 1 : (task == 1 ? g.ntau + 1 : n - k);
    if (col >= ncol) return;
    const int m = task == 0 ? (int)col + 1 : (int)col;
    const cplx Mi = minv_ws[kb];
    const Comp& X = task == 0 ? G.les : (task == 1 ? G.tv : G.ret);
    auto at = [&](int i) { return task == 1 ? (int64_t)i * (g.ntau + 1) + m : tri(i) + m; };
    cplx bdf = cz();
    for (int l = 1; l <= k; ++l) bdf = cadd(bdf, cscal(W.a[l], X.p[at(n - l) * X.ldk + kb]));
    cplx rhs, y;
    if (task == 0) {
        cplx c1, c3, hist;
        const int kv = w.nv == 1 ? 0 : kb;
        hist_les_sums(W, w, G, S.les.p + tri(n) * S.les.ldk, S.les.ldk, w.vec + ((int64_t)w.nv + kv) * w.lenp, n, m, kb, c1,
                      c3, hist);
        const cplx q = csub(cscal(g.h, cmuli(c1)), cscal((double)g.sig * g.htau, c3));
        rhs = cadd(csub(q, cscal(1.0 / g.h, bdf)), cscal(g.h, cmuli(hist)));
        y = cmul(rhs, cconj(Mi));
    } else if (task == 1) {
        rhs = tvq ? q_tv_fft<1>(W, g, G, S, n, m, kb, tvq).v[0][0] : q_tv<1>(W, g, G, S, n, m, kb).v[0][0];
        rhs = csub(csub(rhs, cscal(1.0 / g.h, bdf)), cscal(g.h, cmuli(hist_tv_sum(w, m, kb))));
        y = cmul(Mi, rhs);
    } else {
        rhs = csub(cscal(-1.0 / g.h, bdf), cscal(g.h, cmuli(hist_ret_sum(W, w, G, S, n, m, kb))));
        y = cmul(Mi, rhs);
    }
    if (!cfinite(y)) atomicOr(status, NGF_NONFINITE);
    X.p[at(n) * X.ldk + kb] = y;
}
