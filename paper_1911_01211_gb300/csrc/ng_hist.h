// History sums of a time step by exact digit products on the tensor cores: arguments and host
// interface (kernels: ng_hist.cu; the row vectors and the closing of a step: ng_hist.cuh).
#pragma once

#include "ng_common.cuh"

#define NGH_BLK 128     // rows and columns of a unit of work
#define NGH_PART (2 * NGH_BLK + 1)   // results of a unit and problem
#define NGH_KG 8        // problems of a unit (one warp each)
#define NGH_NVEC 4      // row vectors of a step, see k_hist_vec
#define NGH_DIG_B 1024  // bytes of the digits of 16 elements of a row vector v:
                        // [part][digit][t][half]{Re X, Im X factor}{element 8 half + 2t, + 1} halves,
                        // part 0 (real part of the product): {Re v, -Im v}, part 1: {Im v, Re v}

// Workspace of one step (device pointers).  Units: nbr x nct blocks of the left-mixing rows, then
// the lower block triangles of the lesser and of the retarded history.
struct HistWs {
    cplx* vec;          // [NGH_NVEC][nv][lenp] row vectors with their quadrature weights, FP64
    uint4* tab;         // [NGH_NVEC][nv][lenp/16][64] their digits, see below
    int* vexp;          // [NGH_NVEC][nv][lenp/NGH_BLK] exponent of a block's largest element, -1: a non-finite one
    int* next;          // next unit of work, zeroed by k_hist_vec
    cplx* part;         // [unit][NGH_PART][nb] column sums, row sums, scale of each unit (0: done on the FP64 pipe)
    int nv, lenp;       // problems of the row vectors (1: shared by all), padded length
    int nbr, nct;       // row blocks of the history, column blocks of the left-mixing rows
    int n, T, k, nb;
};

__host__ __device__ __forceinline__ int64_t hist_unit_tv(const HistWs& w, int bi, int bj) {
    return (int64_t)bi * w.nct + bj;
}
__host__ __device__ __forceinline__ int64_t hist_unit_les(const HistWs& w, int bi, int bj) {
    return (int64_t)w.nbr * w.nct + tri(bi) + bj;
}
__host__ __device__ __forceinline__ int64_t hist_unit_ret(const HistWs& w, int bi, int bj) {
    return (int64_t)w.nbr * w.nct + tri(w.nbr) + tri(bi) + bj;
}
__host__ __device__ __forceinline__ int64_t hist_units(const HistWs& w) {
    return (int64_t)w.nbr * w.nct + 2 * tri(w.nbr);
}

// bytes of the workspace for steps up to n_max, and its layout in `base` for step n
size_t hist_ws_bytes(int n_max, int T, int nb, int nv);
HistWs hist_ws_layout(void* base, int n_max, int n, int T, int k, int nb, int nv);
// the column and row sums of every unit into ws.part
cudaError_t hist_launch(const HistWs& ws, const cplx* ret, const cplx* les, const cplx* tv, int sms, int* status,
                        cudaStream_t s);
