// History sums of the uneven batch by digit products: arguments and host interface (products: ng_histu.cu;
// the row vectors and the closing of a step: ng_histu.cuh).
#pragma once

#include "ng_hist.h"

#define NG_UMAXP 128    // problems per launch
struct UProb;

#define NGU_M 128        // free indices of a task
#define NGU_KT 16        // tiles of a task: at least 16, at most 256 (the integer accumulators), 24 tasks to a contraction
#define NGU_CHUNKS 24
#define NGU_SETS 7
#define NGU_NVEC 6

// Sizes of one problem at step n: padded vector length, chunks of a vector (room for them); per set the padded free indices, tiles of a task, chunks of
// the contraction, the first task and the first partial sum; bytes of the problem's part of the workspace.  The
// chunks fall from 24 to 23 and rise again as n grows (the tiles of a task are whole), so the partial sums are laid
// out for the largest number of chunks of any step up to n: no step needs more bytes than a later one, and a
// workspace sized for the last step holds them all.
struct HistUGeo {
    int lenp, vch, free_[NGU_SETS], kt[NGU_SETS], chunks[NGU_SETS], task0[NGU_SETS + 1];
    int64_t poff[NGU_SETS], tab, vexp, conv, part, bytes, slots;   // slots: entries of HistUTab::uexp
};
__host__ __device__ inline void histu_geo(int D, int T, int n, HistUGeo& q) {
    auto pad = [](int64_t x) { return (int)((x + NGU_M - 1) / NGU_M * NGU_M); };
    q.lenp = pad((n > T + 1 ? n : T + 1) * (int64_t)D);
    q.task0[0] = q.vch = 0;
    q.slots = 0;
    int64_t el = 0;
    for (int s = 0; s < NGU_SETS; ++s) {
        const int64_t rows = s >> 1 == 3 ? T + 1 : n, cols = s >> 1 >= 2 ? T + 1 : n, fr = (s & 1) ? rows : cols, con = (s & 1) ? cols : rows;
        q.free_[s] = pad(fr * D);
        const int tiles = (int)((con * D + 15) / 16), kt = (tiles + NGU_CHUNKS - 1) / NGU_CHUNKS;
        q.kt[s] = kt < NGU_KT ? NGU_KT : (kt > 256 ? 256 : kt);
        q.chunks[s] = (tiles + q.kt[s] - 1) / q.kt[s];
        const int most = kt <= NGU_KT || q.chunks[s] > NGU_CHUNKS ? q.chunks[s] : NGU_CHUNKS;
        if (q.vch < most) q.vch = most;
        q.slots += (int64_t)q.free_[s] / NGU_M * most * 8;   // an entry per warp of a task
        q.task0[s + 1] = q.task0[s] + q.free_[s] / NGU_M * q.chunks[s];
        q.poff[s] = el;
        el += (int64_t)q.free_[s] * most * D;
    }
    q.tab = (int64_t)NGU_NVEC * D * q.lenp * sizeof(cplx);
    q.vexp = q.tab + (int64_t)NGU_NVEC * D * (q.lenp / 16) * NGH_DIG_B;
    q.conv = q.vexp + ((int64_t)NGU_NVEC * D * q.vch * (int64_t)sizeof(int) + 255) / 256 * 256;
    q.part = q.conv + (2 * T + 1) * D * D * (int64_t)sizeof(cplx);
    q.bytes = (q.part + el * (int64_t)sizeof(cplx) + 255) / 256 * 256;
}

struct HistUProb {       // written by k_histu_vec
    HermV G, S;
    Grid g;
    cplx* minv;
    cplx* vec;           // [NGU_NVEC][nf][lenp]
    uint4* tab;          // [NGU_NVEC][nf][lenp/16][64]
    int* vexp;           // [NGU_NVEC][nf][vch] exponent of a chunk's largest element, -1: a non-finite one
    cplx* conv;          // Y(i) at i + ntau
    cplx* part;          // per set: [chunk][padded free index][nf]
    HistUGeo q;
};
struct HistUTab {
    HistUProb* probs;    // first in the workspace; a problem's part at base + off[i]
    const UProb* src;
    char* base;
    int *status, *next;   // next task, zeroed by k_histu_vec
    int np, n, ntask;
    int prob[NG_UMAXP], start[NG_UMAXP + 1];   // index into src, first task
    int64_t off[NG_UMAXP];
    int* uexp;             // [task][8] scale of the history of a warp's free indices (0: zeros, or done on the FP64 pipe),
                           // nf at bit 12, problem at bit 16
    int dmax;              // largest nf
};

// rows (time indices) and columns of the matrix of a set; band: j - m above it
struct HistUSet {
    int type, vec, rows, cols, band;   // type 0 retarded, 1 lesser, 2 left-mixing, 3 Matsubara
    bool rowc;                         // rows contracted
};
__device__ __forceinline__ HistUSet histu_set(const Grid& g, int n, int set) {
    HistUSet s;
    s.type = set >> 1;
    s.rowc = (set & 1) == 0;
    s.vec = set == 0 ? 0 : (set == 1 ? 2 : (set == 2 ? 5 : (set >= 5 ? set - 2 : 1)));
    s.rows = s.type == 3 ? g.ntau + 1 : n;
    s.cols = s.type >= 2 ? g.ntau + 1 : n;
    s.band = s.type == 0 || s.type == 3 ? g.k : 0;
    return s;
}
__device__ __forceinline__ const cplx* histu_base(const HistUProb& p, int type) {
    return type == 0 ? p.G.ret.p : (type == 1 ? p.G.les.p : (type == 2 ? p.G.tv.p : p.conv));
}
__device__ __forceinline__ int64_t histu_row(const Grid& g, int type, int j) {
    return type == 3 ? g.ntau - j : (type == 2 ? (int64_t)j * (g.ntau + 1) : tri(j));
}
// tiles of a chunk of a vector: vectors 3 and 4 run over the tau axis, the others over the history
__host__ __device__ __forceinline__ int histu_vec_kt(const HistUGeo& q, int vec) { return q.kt[vec == 3 || vec == 4 ? 5 : 0]; }
// vectors 3 and 5 enter conjugated
__host__ __device__ __forceinline__ bool histu_conj(int vec) { return vec == 3 || vec == 5; }
// last column + 1 of row j in memory
__device__ __forceinline__ int histu_mend(const HistUSet& s, int j) { return s.type >= 2 ? s.cols : max(0, j - s.band); }
// set 6: does the source of column m take row j?
__device__ __forceinline__ bool histu_conv(const HistUSet& s, int ja, int jb, int ma, int mb) {   // all of the ranges
    const int k = s.band, T = s.cols - 1;
    return (ja > mb + k && T - mb > 2 * k + 1) || (jb < ma - k && ma > 2 * k + 1);
}
__device__ __forceinline__ bool histu_has(const HistUSet& s, int j, int m) {
    return j < s.rows && m < histu_mend(s, j) && (s.type != 3 || histu_conv(s, j, j, m, m));
}

// element (j, m) with orbitals: row orbital r, column orbital q (the lesser store holds [column][row])
__device__ __forceinline__ cplx histu_el(const HistUProb& p, const HistUSet& s, int D, int j, int m, int r, int q) {
    return histu_base(p, s.type)[(histu_row(p.g, s.type, j) + m) * D * D + (s.type == 1 ? q * D + r : r * D + q)];
}

// the products of every task into the problems' partial sums
cudaError_t histu_launch(const HistUTab& tab, int sms, cudaStream_t s);
