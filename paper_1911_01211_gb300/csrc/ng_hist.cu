// History sums of a time step on the tensor cores, in exact integer arithmetic.
//
// A step at slice n needs, for every problem, two sums over each stored history element X(j, m):
// the column sum  C(m) = sum_j v(j) X(j, m)  and the row sum  R(j) = sum_m u(m) X(j, m), where v
// and u are row vectors of the step's self-energy slice (ng_hist.cuh says which).  On the FP64
// pipe (2 fused multiply-adds per clock and SM on this part) the sums are bound by arithmetic at
// 2.4 TB/s of history; here every element is read once for both and the products run as f16
// tensor-core products of 8-bit digits, so that the sums are bound by the history's bytes.
//
// Numbers.  X is taken as sign and a 64-bit fixed-point magnitude on the scale 2^E of the largest
// element its warp has met in the unit (E grows in steps of 8 bits, so the window never holds less than
// 56 bits below the largest element), and v as 63 bits on the scale of the largest element of its block of 128:
//   X = +-sum_s d_s 2^(-8(s+1)) 2^(E-1022),  0 <= d_s <= 255,      s = 0..7
//   v =   sum_t q_t 2^(-8(t+1)) 2^(F-1021),  -128 <= q_t <= 128,   t = 0..7
// Products of equal weight u = s + t share an accumulator; the B operand for digit s of X holds the
// digits u - s of v, u = 0..3 in one product (s <= 3) and u = 4..7 in a second, with the real part of
// the complex product in its columns 0..3 and the imaginary part in 4..7.  The contraction index is
// (Re X, Im X) x 8 elements.  Digits of X are encoded as subnormal halves (the byte with the sign
// above it), those of v as integers.  At most 8 * 2 * 32 products of 255 * 128 < 2^15 are added to an
// accumulator before it is moved to a 32-bit integer, so every FP32 accumulation is exact; the result
// is rounded once per unit.  Dropped are the products of weight 8 and more, below 2^-60 of the
// largest product.
//
// Small sums.  All of this is relative to the largest element of the unit, so a sum that is small beside it (the tail
// of a damped function, a column far down the tau axis, a cancellation) would keep fewer bits than on the FP64 pipe.
// With X and v on the scales above, a sum of 128 terms is off by less than 2^-53.8 (the dropped products 2^-54.2, the
// cut of v 2^-56, that of X 2^-57), and by about 2^-60 for errors of random sign.  Where its result is 2^-8 and
// more that is at most 2^-45.8 of it, below the FP64 kernels' bound (256 roundings, 2^-45 of sum |v X|), and 2^-52 for
// random signs, as theirs.  Every sum below 2^-8 whose terms are not all zero is done again on the FP64 pipe
// (k_hist_small), so that no element of a step has less precision than there.
//
// Work.  A unit is 128 x 128 elements of 8 neighbouring problems (128 contiguous bytes per element);
// a warp owns a problem, a ninth warp issues the copies.  16 x 16 tiles of all 8 problems pass through
// a ring of 32 KB stages filled by TMA, one 16-element row per copy, with the 128-byte swizzle: a
// warp reads its problem's 16-byte column without bank conflicts when lanes of odd rows take the
// elements of a pair in the other order.  A warp builds the digits of a tile once, in the layout of
// the A operand with the columns contracted (row sums), and transposes them by movmatrix for the
// column sums.
//
// Measured (512 problems, n = 1600, ntau = 800, 31.5 GB of history): about 8.5 ms, 3.7 TB/s, of a step of 9.4,
// against 28 ms of k_step_bulk, which is bound by the FP64 pipe, of a step of 28.7.  What bounds it is the issue
// of instructions: per tile and warp about 600, and 48 tensor instructions that take 8 issue slots each (mma.sync
// runs at 1024 multiply-adds per clock and SM on this part), with two warps on a scheduler to hide their latency.
#include <cuda.h>

#include "ng_hist.h"

namespace {

constexpr int THREADS = (NGH_KG + 4) * 32;     // eight consumer warps; of the other warpgroup one issues the copies
constexpr int ST = 3;                          // stages of the ring
constexpr int TILE_B = 16 * 16 * NGH_KG * 16;  // history of a stage
constexpr int DIG_B = NGH_DIG_B;               // digits of 16 vector elements
constexpr int U_B = DIG_B + 64;                // and a row of zeros
constexpr int SM_U = ST * TILE_B;              // digits of the row-sum vector: [stage][problem][U_B]
constexpr int SM_COL = SM_U + ST * NGH_KG * U_B;       // column accumulators: [warp][8][2][32] int4
constexpr int SM_ROW = SM_COL + 8 * 16 * 32 * 16;      // row accumulators: [warp][2][32] int4
constexpr int SM_BAR = SM_ROW + 8 * 2 * 32 * 16;       // full[ST], empty[ST]
constexpr int SM_WQ = SM_BAR + 2 * ST * 8;             // work queue: full[2], empty[2], two items
constexpr int SM_BYTES = SM_WQ + 4 * 8 + 2 * 4;
constexpr int E_MIN = 128;                     // smallest scale: everything below 2^-1000 counts as zero
constexpr int WAIT_LIMIT = 1 << 22;            // polls of a barrier before the kernel gives up

struct Args {
    HistWs w;
    const cplx *ret, *les, *tv;
    int64_t nwork;      // units x groups of 8 problems
    int ngrp;
    int* status;
};
struct Maps {           // history as rows of 2 nb doubles
    CUtensorMap tv, les, ret;
};

enum { U_TV = 0, U_LES = 1, U_RET = 2 };

struct Unit {
    int type, bi, bj, grp;
    int64_t id;
};

__device__ __forceinline__ Unit unit_at(const Args& a, int64_t id) {
    Unit u;
    u.id = id;
    u.grp = 0;
    int64_t r = id;
    const int64_t ntv = (int64_t)a.w.nbr * a.w.nct, nt = tri(a.w.nbr);
    if (r < ntv) {
        u.type = U_TV;
        u.bi = (int)(r / a.w.nct);
        u.bj = (int)(r - (int64_t)u.bi * a.w.nct);
        return u;
    }
    r -= ntv;
    u.type = U_LES;
    if (r >= nt) { r -= nt; u.type = U_RET; }
    int b = (int)((sqrtf(8.0f * (float)r + 1.0f) - 1.0f) * 0.5f);
    while (tri(b + 1) <= r) ++b;
    while (tri(b) > r) --b;
    u.bi = b;
    u.bj = (int)(r - tri(b));
    return u;
}
__device__ __forceinline__ Unit unit_of(const Args& a, int64_t wk) {
    Unit u;
    u.id = wk / a.ngrp;
    u.grp = (int)(wk - u.id * a.ngrp);
    int64_t r = u.id;
    const int64_t ntv = (int64_t)a.w.nbr * a.w.nct, nt = tri(a.w.nbr);
    if (r < ntv) {
        u.type = U_TV;
        u.bi = (int)(r / a.w.nct);
        u.bj = (int)(r - (int64_t)u.bi * a.w.nct);
        return u;
    }
    r -= ntv;
    u.type = U_LES;
    if (r >= nt) { r -= nt; u.type = U_RET; }
    int b = (int)((sqrtf(8.0f * (float)r + 1.0f) - 1.0f) * 0.5f);
    while (tri(b + 1) <= r) ++b;
    while (tri(b) > r) --b;
    u.bi = b;
    u.bj = (int)(r - tri(b));
    return u;
}

// columns [m0, m0 + cols) of the strip of 16 rows starting at jr0 that hold any element
__device__ __forceinline__ int strip_cols(const Args& a, const Unit& u, int jr0) {
    const int m0 = u.bj * NGH_BLK;
    int c;
    if (u.type == U_TV) c = a.w.T + 1 - m0;
    else c = min(jr0 + 15, a.w.n - 1) - (u.type == U_RET ? a.w.k : 0) - m0;   // m < j - band
    return max(0, min(c, NGH_BLK));
}

__device__ __forceinline__ int64_t row_offset(const Args& a, int type, int j) {
    return type == U_TV ? (int64_t)j * (a.w.T + 1) : tri(j);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, int bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// false when the phase has not completed within the limit
__device__ __forceinline__ bool mbar_wait(uint32_t bar, int parity) {
#pragma unroll 1
    for (int i = 0; i < WAIT_LIMIT; ++i) {
        uint32_t ok;
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}

// The producer warp: takes items of work from the counter a.w.next, hands them to the consumers through a
// queue of two, and issues the copies of all their tiles in order; lane r < 16 copies row r of the tile, lanes from
// 16 on the row-sum vector's digits of a problem each.  The next item is fetched while the copies of one are issued.
// Items differ in size (triangles and edges hold less): with a fixed share per block the SMs were busy for 81 %
// of a launch for 256 problems, n = 590, ntau = 400; steps 9.89 -> 9.14 ms for 512 problems, n = 1600, ntau = 800,
// 1.42 -> 1.33 ms for 251, n = 777, ntau = 401.
__device__ __forceinline__ void produce(const Args& a, const Maps& maps, uint32_t sbase, int* wq, int lane) {
    const int64_t blk = (int64_t)(a.w.lenp / 16) * DIG_B;   // digits of one vector
    int slot = 0, ph = 1, q = 0, qph = 1;   // an empty stage's first wait passes
    auto give_up = [&] {
        if (lane == 0) atomicOr(a.status, NGF_TIMEOUT);
        for (int i = 0; i < ST; ++i) {   // the copies in flight
            const int sl = (slot + i) % ST;
            mbar_wait(sbase + SM_BAR + sl * 8, sl >= slot ? ph : ph ^ 1);
        }
    };
    int next = lane == 0 ? atomicAdd(a.w.next, 1) : 0;
    while (true) {
        const int wk = __shfl_sync(0xffffffffu, next, 0);
        const bool more = wk < a.nwork;
        if (!mbar_wait(sbase + SM_WQ + 16 + q * 8, qph)) return give_up();
        if (lane == 0) {
            wq[q] = more ? wk : -1;
            mbar_arrive(sbase + SM_WQ + q * 8);
        }
        if (!more) return;
        if (lane == 0) next = atomicAdd(a.w.next, 1);
        if (++q == 2) { q = 0; qph ^= 1; }
        const Unit u = unit_of(a, wk);
        const int k0 = u.grp * NGH_KG, type = u.type, rv = type == U_TV ? 3 : (type == U_LES ? 1 : 2);
        const int ndig = a.w.nv == 1 ? 1 : min(NGH_KG, a.w.nb - k0);
        for (int jr0 = u.bi * NGH_BLK; jr0 < min(u.bi * NGH_BLK + NGH_BLK, a.w.n); jr0 += 16) {
            const int mtn = (strip_cols(a, u, jr0) + 15) >> 4, rows = min(16, a.w.n - jr0);
            for (int mt = 0; mt < mtn; ++mt) {
                const uint32_t full = sbase + SM_BAR + slot * 8, empty = full + ST * 8;
                if (!mbar_wait(empty, ph)) return give_up();
                const int m0 = u.bj * NGH_BLK + mt * 16;
                if (lane == 0) mbar_expect(full, rows * (TILE_B / 16) + ndig * DIG_B);
                __syncwarp();
                if (lane < rows) {
                    const CUtensorMap* map = type == U_TV ? &maps.tv : (type == U_LES ? &maps.les : &maps.ret);
                    const int y = (int)(row_offset(a, type, jr0 + lane) + m0);
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                 ::"r"(sbase + slot * TILE_B + lane * (TILE_B / 16)), "l"(map), "r"(2 * k0), "r"(y), "r"(full)
                                 : "memory");
                } else if (lane >= 16 && lane - 16 < ndig) {
                    const int p = lane - 16;
                    const char* src = (const char*)a.w.tab + ((int64_t)rv * a.w.nv + (a.w.nv == 1 ? 0 : k0 + p)) * blk + (m0 / 16) * DIG_B;
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(sbase + SM_U + (slot * NGH_KG + p) * U_B), "l"(src), "r"(DIG_B), "r"(full)
                                 : "memory");
                }
                __syncwarp();
                if (++slot == ST) { slot = 0; ph ^= 1; }
            }
        }
    }
}

__device__ __forceinline__ void mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t movm(uint32_t x) {
    uint32_t y;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
__device__ __forceinline__ int f2i(float x) { return __float2int_rn(x * 16777216.0f); }
__device__ __forceinline__ uint64_t shr64(uint64_t x, int s) {   // 0 for s >= 64
    uint64_t r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
}

// B operands of the column sums for 16 rows: product i = 0..11 (digit s = i & 3 or i - 4, weights from
// 0 or 4 on) has {Re X, Im X} of rows 0..7, then of rows 8..15 (layout of the table: ng_hist.h).  The
// conjugate vector's digits are the same but for the sign of its imaginary part.
__device__ __forceinline__ void load_digits(uint32_t (&f)[12][4], const uint4* tab, bool conj, int lane) {
    const int g = lane >> 2, t = lane & 3;
    const uint4* p = tab + (g >> 2) * 32 + t;
    const uint32_t x0 = conj && g >= 4 ? 0x80008000u : 0u, x1 = conj && g < 4 ? 0x80008000u : 0u;
#pragma unroll
    for (int i = 0; i < 12; ++i) {
        const int d = i < 4 ? (g & 3) - i : (g & 3) + 8 - i;
        uint4 x = make_uint4(0, 0, 0, 0);
        if (d >= 0) x = __ldg(p + d * 4);
        f[i][0] = x.x ^ x0; f[i][1] = x.y ^ x1; f[i][2] = x.z ^ x0; f[i][3] = x.w ^ x1;
    }
}

// Accumulators of 16 sums: lane (g, t) holds weights 2t, 2t + 1 (t < 2: real part) or 2t - 4, 2t - 3
// (t >= 2: imaginary part) of sum g in .x, .y and of sum g + 8 in .z, .w; lo: weights 0..3, hi: 4..7.
// Their scale grows by 2^(8q): the weights move up by q.
__device__ __forceinline__ void raise(int4& lo, int4& hi, int q) {
    for (; q > 0; --q) {
        const int src = (threadIdx.x & 31) - 1;
        const bool low = (threadIdx.x & 1) == 0;   // t even: weights 0, 1 or 4, 5
        auto step = [&](int& l0, int& l1, int& h0, int& h1) {
            const int pl = __shfl_sync(0xffffffffu, l1, src & 31), ph = __shfl_sync(0xffffffffu, h1, src & 31);
            const int up = __shfl_sync(0xffffffffu, l1, (src + 2) & 31);   // weight 3, from lane t + 1
            h1 = h0;
            h0 = low ? up : ph;
            l1 = l0;
            l0 = low ? 0 : pl;
        };
        step(lo.x, lo.y, hi.x, hi.y);
        step(lo.z, lo.w, hi.z, hi.w);
    }
}
__device__ __forceinline__ int4 to_int(const float (&c)[4]) { return make_int4(f2i(c[0]), f2i(c[1]), f2i(c[2]), f2i(c[3])); }
__device__ __forceinline__ void add(int4& x, const int4 y) { x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w; }

// sum r of stored accumulators [lo, hi][32 lanes]
__device__ __forceinline__ cplx digits_value(const int4* acc, int r, double sc) {
    const int2* p = (const int2*)(acc + 4 * (r & 7)) + (r >> 3);
    double v[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int2 a = p[4 * c], b = p[4 * c + 2], e = p[64 + 4 * c], f = p[64 + 4 * c + 2];
        const long long h = ((long long)a.x << 24) + ((long long)a.y << 16) + ((long long)b.x << 8) + b.y;
        const long long l = ((long long)e.x << 24) + ((long long)e.y << 16) + ((long long)f.x << 8) + f.y;
        v[c] = fma((double)l, 0x1p-32, (double)h) * sc;
    }
    return make_double2(v[0], v[1]);
}
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }

// the sums of one unit and problem on the FP64 pipe: non-finite elements or vectors
__device__ __noinline__ void unit_fp64(const Args& a, const Unit& u, int kb, int cv, int rv, cplx* colp, cplx* rowp,
                                       int lane) {
    const int nb = a.w.nb, n = a.w.n, j0 = u.bi * NGH_BLK, m0 = u.bj * NGH_BLK;
    const int j1 = min(j0 + NGH_BLK, n), band = u.type == U_RET ? a.w.k : 0;
    const cplx* X = (u.type == U_TV ? a.tv : (u.type == U_LES ? a.les : a.ret)) + kb;
    const int kv = a.w.nv == 1 ? 0 : kb;
    const cplx* v = a.w.vec + ((int64_t)cv * a.w.nv + kv) * a.w.lenp;
    const cplx* x = a.w.vec + ((int64_t)rv * a.w.nv + kv) * a.w.lenp;
    auto mend = [&](int j) { return min(m0 + NGH_BLK, u.type == U_TV ? a.w.T + 1 : j - band); };
    for (int c = lane; c < NGH_BLK; c += 32) {
        cplx s = cz();
        for (int j = j0; j < j1; ++j)
            if (m0 + c < mend(j))
                s = cfma(X[(row_offset(a, u.type, j) + m0 + c) * nb], u.type == U_LES ? cconj(v[j]) : v[j], s);
        colp[(int64_t)c * nb] = s;
    }
    for (int r = lane; r < NGH_BLK; r += 32) {
        cplx s = cz();
        if (j0 + r < j1)
            for (int m = m0; m < mend(j0 + r); ++m)
                s = cfma(X[(row_offset(a, u.type, j0 + r) + m) * nb], u.type == U_TV ? cconj(x[m]) : x[m], s);
        rowp[(int64_t)r * nb] = s;
    }
}

__global__ void __launch_bounds__(THREADS, 1) k_hist_mma(const Args a, const __grid_constant__ Maps maps) {
    dep_wait();
    extern __shared__ __align__(1024) unsigned char sm[];
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const unsigned full = 0xffffffffu;
    if (threadIdx.x == 0) {
        for (int i = 0; i < ST; ++i) {
            mbar_init(sbase + SM_BAR + i * 8, 1);
            mbar_init(sbase + SM_BAR + (ST + i) * 8, NGH_KG);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(sbase + SM_WQ + i * 8, 1);
            mbar_init(sbase + SM_WQ + 16 + i * 8, NGH_KG);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < ST * NGH_KG * 4)
        ((uint4*)(sm + SM_U + (threadIdx.x >> 2) * U_B + DIG_B))[threadIdx.x & 3] = make_uint4(0, 0, 0, 0);
    int* wq = (int*)(sm + SM_WQ + 32);
    __syncthreads();
    // registers of the launch: 12 x 32 x 168; the consumers take 224, the others keep 40
    if (warp >= NGH_KG) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == NGH_KG) produce(a, maps, sbase, wq, lane);
        return;
    }
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    int4* colacc = (int4*)(sm + SM_COL) + warp * 16 * 32;
    int4* rowacc = (int4*)(sm + SM_ROW) + warp * 2 * 32;
    int slot = 0, ph = 0;
    // this lane's elements: rows g, g + 8, columns 2t, 2t + 1, 2t + 8, 2t + 9; lanes of odd rows load the
    // columns of a pair in the other order (their lines then lie in other banks)
    const uint32_t l0 = (uint32_t)(g * 2048 + (2 * t + (g & 1)) * 128 + ((warp ^ (2 * t + (g & 1))) << 4));
    const uint32_t l1 = (uint32_t)(g * 2048 + (2 * t + (~g & 1)) * 128 + ((warp ^ (2 * t + (~g & 1))) << 4));
    const uint32_t pack_hi = g & 1 ? 0x3276u : 0x7632u, pack_lo = g & 1 ? 0x1054u : 0x5410u;
    // digit (g & 3) - i of the row-sum vector, i = 0..3; none below 0
    int uo[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        uo[i] = SM_U + warp * (a.w.nv == 1 ? 0 : U_B) + ((g & 3) >= i ? (g >> 2) * 512 + ((g & 3) - i) * 64 : DIG_B) + t * 16;

#pragma unroll 1
    for (int q = 0, qph = 0;;) {
        if (!mbar_wait(sbase + SM_WQ + q * 8, qph)) {
            if (lane == 0) atomicOr(a.status, NGF_TIMEOUT);
            return;
        }
        const int wk = ((volatile int*)wq)[q];
        __syncwarp();
        if (lane == 0) mbar_arrive(sbase + SM_WQ + 16 + q * 8);
        if (++q == 2) { q = 0; qph ^= 1; }
        if (wk < 0) return;
        const Unit u = unit_of(a, wk);
        const int kb = u.grp * NGH_KG + warp;
        const bool act = kb < a.w.nb;
        const int kv = a.w.nv == 1 ? 0 : min(kb, a.w.nb - 1);
        const int j0 = u.bi * NGH_BLK, m0 = u.bj * NGH_BLK, jend = min(j0 + NGH_BLK, a.w.n);
        const int band = u.type == U_RET ? a.w.k : 0;
        const int cv = u.type == U_RET ? 0 : 1, rv = u.type == U_TV ? 3 : (u.type == U_LES ? 1 : 2);
        const uint4* ctab = a.w.tab + (((int64_t)cv * a.w.nv + kv) * (a.w.lenp / 16) + j0 / 16) * (DIG_B / 16);
        const int nblk = a.w.lenp / NGH_BLK;
        const int fc = a.w.vexp[(cv * a.w.nv + kv) * nblk + u.bi], fr = a.w.vexp[(rv * a.w.nv + kv) * nblk + u.bj];
        cplx* colp = a.w.part + u.id * NGH_PART * a.w.nb + kb;
        cplx* rowp = colp + (int64_t)NGH_BLK * a.w.nb;
        bool bad = fc < 0 || fr < 0;
        int E = 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) colacc[i * 32 + lane] = make_int4(0, 0, 0, 0);
#pragma unroll 1
        for (int jr0 = j0; jr0 < jend; jr0 += 16) {
            const int mtn = (strip_cols(a, u, jr0) + 15) >> 4;
            uint32_t va[12][4];
            load_digits(va, ctab + ((jr0 - j0) / 16) * (DIG_B / 16), u.type == U_LES, lane);
            float rlo[4] = {0.f, 0.f, 0.f, 0.f}, rhi[4] = {0.f, 0.f, 0.f, 0.f};
            int4 ilo = make_int4(0, 0, 0, 0), ihi = ilo;
#pragma unroll 1
            for (int mt = 0; mt < mtn; ++mt) {
                if (!mbar_wait(sbase + SM_BAR + slot * 8, ph)) {
                    if (lane == 0) atomicOr(a.status, NGF_TIMEOUT);
                    return;
                }
                const unsigned char* p = sm + slot * TILE_B;
                const unsigned char* up = sm + slot * NGH_KG * U_B;
                const uint32_t empty = sbase + SM_BAR + (ST + slot) * 8;
                if (++slot == ST) { slot = 0; ph ^= 1; }
                if (!act) {
                    if (lane == 0) mbar_arrive(empty);
                    continue;
                }
                uint32_t h[2][4][2], l[2][4][2];   // [row g + 8 jh][column][re, im]
#pragma unroll
                for (int jh = 0; jh < 2; ++jh)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint4 x = *(const uint4*)(p + ((i & 1) ? l1 : l0) + jh * 16384 + (i >> 1) * 1024);
                        l[jh][i][0] = x.x; h[jh][i][0] = x.y; l[jh][i][1] = x.z; h[jh][i][1] = x.w;
                    }
                const int jt = jr0, mt0 = m0 + mt * 16;
                if (jt + 16 > a.w.n || (u.type == U_TV ? mt0 + 15 > a.w.T : mt0 + 15 >= jt - band)) {
                    // tile at an edge: elements outside the history or in the band count as zero
#pragma unroll
                    for (int jh = 0; jh < 2; ++jh)
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int j = jt + g + 8 * jh, m = mt0 + 2 * t + ((g ^ i) & 1) + (i >> 1) * 8;
                            if (j >= a.w.n || m > (u.type == U_TV ? a.w.T : j - band - 1)) h[jh][i][0] = h[jh][i][1] = 0;
                        }
                }
                int sh[2][4][2];
                int neg = 0;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const uint32_t x = (&h[0][0][0])[i];
                    neg |= (&sh[0][0][0])[i] = E - (int)((x + x) >> 21);
                }
                if (E == 0 || __any_sync(full, neg < 0)) {   // first tile, or a larger element: raise the scale
                    int lo = 0;
#pragma unroll
                    for (int i = 0; i < 16; ++i) lo = min(lo, (&sh[0][0][0])[i]);
                    const int emax = E + __reduce_max_sync(full, -lo);
                    bad = bad || emax == 2047;
                    int dE;
                    if (E == 0) dE = max(emax + 1, E_MIN);   // a bit of room: the parts of a value that turns grow by up to sqrt(2)
                    else {
                        const int q = (emax - E + 7) >> 3, qs = min(q, 8);
                        dE = 8 * q;
                        add(ilo, to_int(rlo));
                        add(ihi, to_int(rhi));
                        raise(ilo, ihi, qs);
#pragma unroll
                        for (int i = 0; i < 4; ++i) rlo[i] = rhi[i] = 0.f;
#pragma unroll 1
                        for (int i = 0; i < 8; ++i) {
                            int4 x = colacc[(2 * i) * 32 + lane], y = colacc[(2 * i + 1) * 32 + lane];
                            raise(x, y, qs);
                            colacc[(2 * i) * 32 + lane] = x;
                            colacc[(2 * i + 1) * 32 + lane] = y;
                        }
                    }
                    E += dE;
#pragma unroll
                    for (int i = 0; i < 16; ++i) (&sh[0][0][0])[i] += dE;
                }
                // 16-bit chunks of the magnitudes of each pair of columns (2t, 2t+1 | 2t+8, 2t+9), and
                // their signs at bits 15 and 31
                uint32_t P[2][2][2][4], S[2][2][2];   // [jh][mh][re, im]
#pragma unroll
                for (int jh = 0; jh < 2; ++jh)
#pragma unroll
                    for (int mh = 0; mh < 2; ++mh)
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            uint32_t xh[2], xl[2];
#pragma unroll
                            for (int z = 0; z < 2; ++z) {
                                const int i = 2 * mh + z;
                                const uint32_t top = __funnelshift_l(l[jh][i][c], h[jh][i][c], 11) | 0x80000000u;
                                const uint64_t M = shr64(((uint64_t)top << 32) | (l[jh][i][c] << 11), sh[jh][i][c]);
                                xh[z] = (uint32_t)(M >> 32);
                                xl[z] = (uint32_t)M;
                            }
                            P[jh][mh][c][0] = __byte_perm(xh[0], xh[1], pack_hi);
                            P[jh][mh][c][1] = __byte_perm(xh[0], xh[1], pack_lo);
                            P[jh][mh][c][2] = __byte_perm(xl[0], xl[1], pack_hi);
                            P[jh][mh][c][3] = __byte_perm(xl[0], xl[1], pack_lo);
                            S[jh][mh][c] = __byte_perm(h[jh][2 * mh][c], h[jh][2 * mh + 1][c], pack_hi) & 0x80008000u;
                        }
                float clo[4] = {0.f, 0.f, 0.f, 0.f}, chi[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    uint32_t d[2][2][2], e[2][2][2];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        (&d[0][0][0])[i] = __byte_perm((&P[0][0][0][0])[i * 4 + (s >> 1)], (&S[0][0][0])[i], (s & 1) ? 0x7250 : 0x7351);
                        (&e[0][0][0])[i] = movm((&d[0][0][0])[i]);
                    }
#pragma unroll
                    for (int hi = s < 4 ? 0 : 1; hi < 2; ++hi) {
                        const int i = s - 4 * hi;   // digit (g & 3) - i of the vector
                        const uint4 x = *(const uint4*)(up + (i <= 0 ? uo[0] - i * 64 : uo[i > 0 ? i : 0]));
                        float(&R)[4] = hi ? rhi : rlo;
                        float(&C)[4] = hi ? chi : clo;
                        const uint32_t(&v)[4] = va[hi ? 4 + s : s];
                        mma(R, d[0][0][0], d[1][0][0], d[0][0][1], d[1][0][1], x.x, x.y);
                        mma(C, e[0][0][0], e[0][1][0], e[0][0][1], e[0][1][1], v[0], v[1]);
                        mma(R, d[0][1][0], d[1][1][0], d[0][1][1], d[1][1][1], x.z, x.w);
                        mma(C, e[1][0][0], e[1][1][0], e[1][0][1], e[1][1][1], v[2], v[3]);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(empty);
                int4* z = colacc + mt * 64 + lane;
                int4 v = z[0];
                add(v, to_int(clo));
                z[0] = v;
                v = z[32];
                add(v, to_int(chi));
                z[32] = v;
                if ((mt & 1) || mt == mtn - 1) {   // 32 columns added
                    add(ilo, to_int(rlo));
                    add(ihi, to_int(rhi));
#pragma unroll
                    for (int i = 0; i < 4; ++i) rlo[i] = rhi[i] = 0.f;
                }
            }
            if (!act) continue;
            rowacc[lane] = ilo;
            rowacc[32 + lane] = ihi;
            __syncwarp();
            const double sc = bad ? 0.0 : pow2(max(E, E_MIN) - 1022 - 20) * pow2(fr - 1021 - 20);
            if (lane < 16) rowp[(int64_t)(jr0 - j0 + lane) * a.w.nb] = digits_value(rowacc, lane, sc);
            __syncwarp();
        }
        if (!act) continue;
        __syncwarp();
        if (lane == 0) rowp[(int64_t)NGH_BLK * a.w.nb].x = bad ? 0.0 : E;
        const double sc = bad ? 0.0 : pow2(max(E, E_MIN) - 1022 - 20) * pow2(fc - 1021 - 20);
        for (int i = lane; i < NGH_BLK; i += 32) colp[(int64_t)i * a.w.nb] = digits_value(colacc + (i >> 4) * 64, i & 15, sc);
        __syncwarp();
        if (bad) unit_fp64(a, u, kb, cv, rv, colp, rowp, lane);   // a non-finite element or vector
    }
}

// The sums that are small on the scale of their unit, again on the FP64 pipe.  A warp takes SMALL_Q sums of 32
// neighbouring problems at a time: it reads the results, whole lines, compares their exponents with the scales, and does
// the small ones four at once, eight lanes to a sum (70 FP64 instructions for the four, which bound the kernel where many
// are small; else it is the read of the results).  In a kernel of its own because small sums lie in a few problems, and
// the ring of k_hist_mma goes at the pace of its slowest warp: done there, 0.2 % of the sums took the step of 251
// problems, n = 777, ntau = 401 from 1.28 to 2.18 ms.  Here, of whole steps: 512 problems, n = 1600, ntau = 800 (0.02 % of
// the sums) 0.16 ms of 9.4; the 251 problems 0.06 of 1.36; 256 problems, n = 900, ntau = 400 (0.6 %) 0.08 of 1.76; a
// second-Born run of 128 problems, n = 160, ntau = 200 (8 %, most of them columns far down the tau axis) 106 -> 115 ms.
template <int SMALL_Q>
__global__ void __launch_bounds__(128) k_hist_small(const Args a) {
    dep_wait();
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, nb = a.w.nb, nkb = (nb + 31) / 32, nblk = a.w.lenp / NGH_BLK;
    const int64_t items = hist_units(a.w) * (2 * NGH_BLK / SMALL_Q) * nkb, step = (int64_t)gridDim.x * blockDim.x >> 5;
    for (int64_t it = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += step) {
        const int64_t r = it / nkb, id = r / (2 * NGH_BLK / SMALL_Q);
        const int kb0 = (int)(it - r * nkb) * 32, kb = min(kb0 + lane, nb - 1), i0 = (int)(r % (2 * NGH_BLK / SMALL_Q)) * SMALL_Q;
        const bool row = i0 >= NGH_BLK;
        cplx* p = a.w.part + (id * NGH_PART + i0) * nb;
        const int E = (int)p[(int64_t)(2 * NGH_BLK - i0) * nb + kb].x;
        int ex[SMALL_Q];
#pragma unroll
        for (int q = 0; q < SMALL_Q; ++q) {
            const cplx x = p[(int64_t)q * nb + kb];
            ex[q] = max(__double2hiint(x.x) >> 20 & 2047, __double2hiint(x.y) >> 20 & 2047);
        }
        const Unit u = unit_at(a, id);
        const int vec = row ? (u.type == U_TV ? 3 : (u.type == U_LES ? 1 : 2)) : (u.type == U_RET ? 0 : 1);
        const int F = a.w.vexp[(vec * a.w.nv + (a.w.nv == 1 ? 0 : kb)) * nblk + (row ? u.bj : u.bi)];
        const int low = max(E + F - 2043 - 8 + 1023, 1);   // exponent of 2^-8 on the scale 2^(E-1022) 2^(F-1021)
        const int j0 = u.bi * NGH_BLK, m0 = u.bj * NGH_BLK, j1 = min(j0 + NGH_BLK, a.w.n), band = u.type == U_RET ? a.w.k : 0;
        // terms [c0, c1) of sum i0 + q: row j0 + i over its columns, or column m0 + i over its rows
        auto range = [&](int q, int& c0, int& c1) {
            const int i = (i0 + q) % NGH_BLK;
            if (row) {
                c0 = m0;
                c1 = j0 + i >= j1 ? 0 : min(m0 + NGH_BLK, u.type == U_TV ? a.w.T + 1 : j0 + i - band);
            } else {
                c0 = u.type == U_TV ? j0 : max(j0, m0 + i + band + 1);
                c1 = u.type == U_TV && m0 + i > a.w.T ? 0 : j1;
            }
        };
        unsigned left[SMALL_Q];
        int total = 0;
#pragma unroll
        for (int q = 0; q < SMALL_Q; ++q) {
            int c0, c1;
            range(q, c0, c1);
            // scales above E_MIN: neither the history's unit nor the vector's block is zero
            left[q] = __ballot_sync(full, kb0 + lane < nb && E > E_MIN && F > E_MIN && ex[q] < low && c0 < c1);
            total += __popc(left[q]);
        }
        const bool conj = u.type == (row ? U_TV : U_LES);
        const cplx* X = u.type == U_TV ? a.tv : (u.type == U_LES ? a.les : a.ret);
        for (int base = 0; base < total; base += 4) {
            int at = base + (lane >> 3), q = 0;   // this group's sum: the at-th of the masks in turn
            const bool mine = at < total;
            if (!mine) at = total - 1;
            while (q < SMALL_Q - 1 && at >= __popc(left[q])) at -= __popc(left[q++]);
            const int k = kb0 + (int)__fns(left[q], 0, at + 1), i = (i0 + q) % NGH_BLK;
            int c0, c1;
            range(q, c0, c1);
            const cplx* v = a.w.vec + ((int64_t)vec * a.w.nv + (a.w.nv == 1 ? 0 : k)) * a.w.lenp;
            cplx s = cz();
#pragma unroll 4
            for (int c = c0 + (lane & 7); c < c1; c += 8) {
                const int64_t el = row ? row_offset(a, u.type, j0 + i) + c : row_offset(a, u.type, c) + m0 + i;
                s = cfma(X[el * nb + k], conj ? cconj(v[c]) : v[c], s);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                s.x += __shfl_xor_sync(full, s.x, o);
                s.y += __shfl_xor_sync(full, s.y, o);
            }
            if (mine && (lane & 7) == 0) p[(int64_t)q * nb + k] = s;
        }
    }
}

inline int pad_blk(int x) { return (x + NGH_BLK - 1) / NGH_BLK * NGH_BLK; }
inline size_t up256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

static HistWs layout(char* base, int n_max, int n, int T, int k, int nb, int nv, size_t* bytes) {
    HistWs w;
    w.n = n; w.T = T; w.k = k; w.nb = nb; w.nv = nv;
    w.lenp = pad_blk(n_max > T + 1 ? n_max : T + 1);
    w.nct = pad_blk(T + 1) / NGH_BLK;
    size_t o = 0;
    w.vec = (cplx*)(base + o);
    o += up256(sizeof(cplx) * (size_t)NGH_NVEC * nv * w.lenp);
    w.tab = (uint4*)(base + o);
    o += up256((size_t)NGH_NVEC * nv * (w.lenp / 16) * DIG_B);
    w.vexp = (int*)(base + o);
    o += up256(sizeof(int) * (size_t)NGH_NVEC * nv * (w.lenp / NGH_BLK));
    w.next = (int*)(base + o);
    o += 256;
    w.part = (cplx*)(base + o);
    w.nbr = pad_blk(n_max) / NGH_BLK;
    o += sizeof(cplx) * (size_t)hist_units(w) * NGH_PART * nb;
    w.nbr = pad_blk(n) / NGH_BLK;
    if (bytes) *bytes = o;
    return w;
}

size_t hist_ws_bytes(int n_max, int T, int nb, int nv) {
    size_t b;
    layout(nullptr, n_max, n_max, T, 1, nb, nv, &b);
    return b;
}

HistWs hist_ws_layout(void* base, int n_max, int n, int T, int k, int nb, int nv) {
    return layout((char*)base, n_max, n, T, k, nb, nv, nullptr);
}

// 2D map of `rows` history elements of nb problems: boxes of 16 elements x 8 problems, swizzled
static bool make_map(CUtensorMap* m, const cplx* p, int64_t rows, int nb) {
    typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                               const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static Encode encode = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return (Encode)f;
    }();
    const cuuint64_t dims[2] = {(cuuint64_t)2 * nb, (cuuint64_t)rows}, strides[1] = {(cuuint64_t)nb * sizeof(cplx)};
    const cuuint32_t box[2] = {2 * NGH_KG, 16}, one[2] = {1, 1};
    return encode && encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, (void*)p, dims, strides, box, one,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t hist_launch(const HistWs& ws, const cplx* ret, const cplx* les, const cplx* tv, int sms, int* status,
                        cudaStream_t s) {
    Args a;
    a.w = ws;
    a.ret = ret;
    a.les = les;
    a.tv = tv;
    a.status = status;
    a.ngrp = (ws.nb + NGH_KG - 1) / NGH_KG;
    a.nwork = hist_units(ws) * a.ngrp;
    Maps maps;
    if (!make_map(&maps.tv, tv, (int64_t)ws.n * (ws.T + 1), ws.nb) || !make_map(&maps.les, les, tri(ws.n), ws.nb) ||
        !make_map(&maps.ret, ret, tri(ws.n), ws.nb))
        return cudaErrorNotSupported;
    cudaError_t e = cudaFuncSetAttribute(k_hist_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, SM_BYTES);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)(a.nwork < sms ? a.nwork : sms);
    dep_launch(k_hist_mma, grid, THREADS, SM_BYTES, s)(a, maps);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // sums of 32 problems; one at a time while these are fewer than four for each warp the GPU holds
    const int64_t sums = hist_units(ws) * 2 * NGH_BLK * ((ws.nb + 31) / 32);
    const unsigned most = 16 * (unsigned)sms;
    if (sums < 16 * (int64_t)most) dep_launch(k_hist_small<1>, (unsigned)(sums < 4 * (int64_t)most ? (sums + 3) / 4 : most), 128, 0, s)(a);
    else dep_launch(k_hist_small<4>, most, 128, 0, s)(a);
    return cudaGetLastError();
}
