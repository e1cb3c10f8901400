// History sums of the uneven batch (problems of 1, 2, 4 or 8 orbitals, each with its own storage) by
// exact digit products on the tensor cores; numbers and digits as in ng_hist.cu, with a scale of X for a warp's 16 free
// indices in a task, of a vector for each chunk of the contraction.  A sum below 2^-8 on these scales (a weak
// coupling between orbitals, a damped tail, a cancellation) is done again on the FP64 pipe, for the reason given there
// (its bounds are per term, those of the FP64 kernels too).
//
// With orbitals the stored history of a component is a matrix X over (time, orbital) pairs, and the
// sums of a step are products of X or its transpose with nf row vectors each (vectors: k_histu_vec):
//   set 0  retarded, rows contracted     ret item m, (a, b): sum v0_a (j c) X^R(j, m)[c b]
//   set 1  retarded, columns contracted  C^<_1 of row j:     sum X^R(j, m)[a c] v2_b (m c)
//   set 2  lesser, rows contracted       history of m, l > m: sum conj(v5_b (l c)) X^<(m, l)[a c], v5 = v1
//   set 3  lesser, columns contracted    history of l, m < l: -conj(sum v1_b (m c) X^<(m, l)[c a])
//   set 4  left-mixing, rows contracted  tv item m:          sum v1_a (j c) X(j, m)[c b]
//   set 5  left-mixing, columns contracted  C^<_3 of row j:  sum X(j, m)[a c] v3_b (m c)
//   set 6  Matsubara source of tv item m:   sum v4_a (j c) Y(m - j)[c b], |j - m| > k, where Y(i) is G^M(-i)
//          for i < 0 and xi G^M(ntau - i) for i > 0; the convolution over [0, m] only where m > 2k + 1, that
//          over [m, ntau] only where ntau - m > 2k + 1
// The FP64 pipe does them in about 4 n (n + ntau) nf^3 complex multiply-adds at one per 2 clocks and SM.
// Here a task is 128 free indices (16 a warp, M of the product) and at least 16 tiles of 16 contracted
// ones; a ninth warp copies a tile's rows (contiguous in one problem's storage) into a ring by
// cp.async.bulk.  Each warp turns its 16 x 16 elements into digits once and multiplies them with the
// digits of all nf vectors, so the conversion (about 400 issue slots a tile) is paid once for nf x 24 tensor
// instructions of 8 slots; the two directions are separate tasks, which reads X twice but needs no
// transposition and keeps no column sums.
//
// Measured (16 clusters, one of 8, four of 4, five of 2 orbitals, n = 500, ntau = 300): 1.14 ms (1.31 with a fixed
// share of tasks per block), with k_histu_close 0.19, k_histu_small 0.22 and k_histu_vec 0.02 against 6.3 ms of k_ubulk.  The issue slots alone are 0.6 ms; the
// rest is shared memory (per tile and output 8 loads of 512 bytes of digits, and the elements, whose
// orbital stride of 128 bytes at nf = 8 puts four lanes of eight on one bank in half the sets) and the
// latency of two warps per quarter of an SM.
#include "ng_histu.h"

namespace {

constexpr int THREADS = 384, ST = 3;
constexpr int TILE_B = 32768 + 2048;                 // 16 x 128 elements, rows padded by 16 bytes
constexpr int U_B = NGH_DIG_B + 64;                  // digits of a vector, a row of zeros
constexpr int SM_U = ST * TILE_B;                    // [stage][output][U_B]
constexpr int SM_INT = SM_U + ST * 8 * U_B;          // integer accumulators: [warp][output][lo, hi][32] int4
constexpr int SM_BAR = SM_INT + 8 * 8 * 2 * 32 * 16;
constexpr int SM_WQ = SM_BAR + 2 * ST * 8;             // task queue: full[2], empty[2], two tasks
constexpr int SM_TASK = SM_WQ + 4 * 8 + 2 * 4;         // the task of each warp
constexpr int SM_BYTES = SM_TASK + 8 * 4;

struct Task {
    const HistUProb* p;
    HistUSet s;
    int D, set, chunk, f0, kt0, kt1;   // free indices from f0; contracted tiles [kt0, kt1)
};

// task tk; kt1 <= kt0 when the history has no element there
__device__ __forceinline__ Task task_at(const HistUTab& tab, int tk, int i) {   // of problem i
    Task t;
    t.p = &tab.probs[i];
    int r = tk - tab.start[i];
    t.set = 0;
    while (r >= t.p->q.task0[t.set + 1]) ++t.set;
    r -= t.p->q.task0[t.set];
    const int nm = t.p->q.free_[t.set] / NGU_M;
    t.chunk = r / nm;
    t.f0 = (r % nm) * NGU_M;
    t.D = t.p->g.nf;
    t.s = histu_set(t.p->g, tab.n, t.set);
    const int ncon = (t.s.rowc ? t.s.rows : t.s.cols) * t.D;
    t.kt0 = t.chunk * t.p->q.kt[t.set];
    t.kt1 = min(t.kt0 + t.p->q.kt[t.set], (ncon + 15) / 16);
    if (t.s.type < 2) {
        if (t.s.rowc) t.kt0 = max(t.kt0, (t.f0 / t.D + t.s.band + 1) * t.D / 16);           // rows j > m + band
        else {
            const int jl = min((t.f0 + NGU_M - 1) / t.D, t.s.rows - 1);                      // columns m < j - band
            t.kt1 = min(t.kt1, (max(0, jl - t.s.band) * t.D + 15) / 16);
        }
    }
    return t;
}

__device__ __forceinline__ Task task_of(const HistUTab& tab, int tk) {
    int i = 0;
    while (tk >= tab.start[i + 1]) ++i;
    return task_at(tab, tk, i);
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
__device__ __forceinline__ bool mbar_wait(uint32_t bar, int parity) {
#pragma unroll 1
    for (int i = 0; i < (1 << 22); ++i) {
        uint32_t ok;
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void bulk(uint32_t dst, const void* src, int bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
                 "r"(bytes), "r"(bar) : "memory");
}

// Time rows of a tile step and their columns: rows contracted: JT rows x 128/D columns from f0; columns
// contracted: 128/D rows x JT columns.  Row i of the tile lies at i * (cols D^2 16 + 16) bytes.
struct Span { int j0, nj, m0, nm; };
__device__ __forceinline__ Span span_of(const Task& t, int kt) {
    const int JT = 16 / t.D, F = NGU_M / t.D;
    Span s;
    if (t.s.rowc) { s.j0 = kt * JT; s.nj = JT; s.m0 = t.f0 / t.D; s.nm = F; }
    else { s.j0 = t.f0 / t.D; s.nj = F; s.m0 = kt * JT; s.nm = JT; }
    return s;
}

// The producer warp; tasks, which differ by the orbitals and the triangles, come from a counter as in ng_hist.cu
__device__ __forceinline__ void produce(const HistUTab& tab, uint32_t sbase, int* wq, int lane) {
    int slot = 0, ph = 1, w = 0, wph = 1;
    auto give_up = [&] {
        if (lane == 0) atomicOr(tab.status, NGF_TIMEOUT);
        for (int i = 0; i < ST; ++i) {   // the copies in flight
            const int sl = (slot + i) % ST;
            mbar_wait(sbase + SM_BAR + sl * 8, sl >= slot ? ph : ph ^ 1);
        }
    };
    int next = lane == 0 ? atomicAdd(tab.next, 1) : 0;
    while (true) {
        const int tk = __shfl_sync(0xffffffffu, next, 0);
        const bool more = tk < tab.ntask;
        if (!mbar_wait(sbase + SM_WQ + 16 + w * 8, wph)) return give_up();
        if (lane == 0) {
            wq[w] = more ? tk : -1;
            mbar_arrive(sbase + SM_WQ + w * 8);
        }
        if (!more) return;
        if (lane == 0) next = atomicAdd(tab.next, 1);
        if (++w == 2) { w = 0; wph ^= 1; }
        const Task t = task_of(tab, tk);
        const int D = t.D, DD16 = D * D * 16;
        const char* base = (const char*)histu_base(*t.p, t.s.type);
        for (int kt = t.kt0; kt < t.kt1; ++kt) {
            const uint32_t full = sbase + SM_BAR + slot * 8, empty = full + ST * 8;
            if (!mbar_wait(empty, ph)) return give_up();
            const Span s = span_of(t, kt);
            auto bytes_of = [&](int i) {   // stored elements of row j0 + i inside the span
                const int j = s.j0 + i;
                if (i >= s.nj || j >= t.s.rows) return 0;
                return max(0, min(s.nm, histu_mend(t.s, j) - s.m0)) * DD16;
            };
            int b = 0;
            for (int i = lane; i < s.nj; i += 32) b += bytes_of(i);
            b = __reduce_add_sync(0xffffffffu, b);
            if (lane == 0) mbar_expect(full, b + D * NGH_DIG_B);
            __syncwarp();
            const uint32_t st = sbase + slot * TILE_B;
            for (int i = lane; i < s.nj; i += 32)
                if (const int x = bytes_of(i))
                    bulk(st + i * (s.nm * DD16 + 16), base + (histu_row(t.p->g, t.s.type, s.j0 + i) + s.m0) * DD16, x, full);
            if (lane < D)
                bulk(sbase + SM_U + (slot * 8 + lane) * U_B,
                     (const char*)t.p->tab + (((int64_t)t.s.vec * D + lane) * (t.p->q.lenp / 16) + kt) * NGH_DIG_B, NGH_DIG_B, full);
            __syncwarp();
            if (++slot == ST) { slot = 0; ph ^= 1; }
        }
    }
}

__device__ __forceinline__ void mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint64_t shr64(uint64_t x, int s) {   // 0 for s >= 64
    uint64_t r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
}
__device__ __forceinline__ int f2i(float x) { return __float2int_rn(x * 16777216.0f); }
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }
// the 16 sums of accumulators (lane (g, t): weights 2t.. of sums g, g + 8), one number per lane: sum
// g + 8 (t & 1), real part for t < 2
__device__ __forceinline__ double digits_value(int4 lo, int4 hi, double sc) {
    const bool low = (threadIdx.x & 1) == 0;
    auto pair = [&](int x, int y) { const long long v = ((long long)x << 8) + y; return low ? v << 16 : v; };
    const long long h0 = pair(lo.x, lo.y), l0 = pair(hi.x, hi.y), h1 = pair(lo.z, lo.w), l1 = pair(hi.z, hi.w);
    const long long h = __shfl_xor_sync(0xffffffffu, low ? h1 : h0, 1) + (low ? h0 : h1);
    const long long l = __shfl_xor_sync(0xffffffffu, low ? l1 : l0, 1) + (low ? l0 : l1);
    return fma((double)l, 0x1p-32, (double)h) * sc;
}

__device__ __forceinline__ bool nonzero(cplx x) {   // on the integer pipe
    return ((unsigned)(__double2hiint(x.x) << 1) | (unsigned)__double2loint(x.x) | (unsigned)(__double2hiint(x.y) << 1) |
            (unsigned)__double2loint(x.y)) != 0;
}
// contracted times [lo, hi) of free time f in a task (all that the matrix holds; set 6 has gaps)
__device__ __forceinline__ void task_range(const Task& t, int f, int& lo, int& hi) {
    const HistUSet& s = t.s;
    lo = t.kt0 * 16 / t.D;
    hi = min(t.kt1 * 16 / t.D, s.rowc ? s.rows : s.cols);
    if (f >= (s.rowc ? s.cols : s.rows)) hi = 0;
    else if (s.type < 2) {
        if (s.rowc) lo = max(lo, f + s.band + 1);
        else hi = min(hi, histu_mend(s, f));
    }
}

// The sums that are small on their scale, again on the FP64 pipe, in a kernel of its own as in ng_hist.cu: a warp takes
// 16 free indices and an output of a task and does the small sums four at once, eight lanes to a sum, four terms of a lane
// in flight; terms whose couplings are zero cost no arithmetic.  Whole steps without and with it: 16 clusters of 1 to 8
// orbitals, n = 500, ntau = 300 1.87 / 2.05 ms; one of 8, n = 250, ntau = 60 (no small sums) 0.65 / 0.67.
__global__ void __launch_bounds__(128) k_histu_small(const __grid_constant__ HistUTab tab) {
    dep_wait();
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < tab.ntask * 8 * tab.dmax; i += gridDim.x * blockDim.x >> 5) {
        const int tw = i / tab.dmax, o = i - tw * tab.dmax, code = tab.uexp[tw], E = code & 0xfff, D = code >> 12 & 15;
        if (E <= 128 || o >= D) continue;
        const Task t = task_at(tab, tw >> 3, code >> 16);
        const HistUSet& s = t.s;
        const int f0 = t.f0 + (tw & 7) * 16;
        cplx* out = t.p->part + t.p->q.poff[t.set] + ((int64_t)t.chunk * t.p->q.free_[t.set] + f0) * D + o;
        const int F = t.p->vexp[(s.vec * D + o) * t.p->q.vch + t.chunk];
        bool is = false;
        if (lane < 16) {
            const cplx x = out[lane * D];
            int lo, hi;
            task_range(t, (f0 + lane) / D, lo, hi);
            // 2^-8 on the scale 2^(E-1022) 2^(F-1021); scales of 128: zeros
            const int ex = max(__double2hiint(x.x) >> 20 & 2047, __double2hiint(x.y) >> 20 & 2047);
            is = lo < hi && F > 128 && ex < max(E + F - 2043 - 8 + 1023, 1);
        }
        const cplx* v = t.p->vec + ((int64_t)s.vec * D + o) * t.p->q.lenp;
        for (unsigned left = __ballot_sync(full, is); left;) {
            unsigned rest = left;   // this group's sum: the bit number lane / 8, else the first
            for (int z = lane >> 3; z > 0; --z) rest &= rest - 1;
            const bool mine = rest != 0;
            const int r = __ffs(mine ? rest : left) - 1, f = (f0 + r) / D, fo = (f0 + r) % D;
            for (int z = 0; z < 4; ++z) left &= left - 1;
            int lo, hi;
            task_range(t, f, lo, hi);
            const int steps = (__reduce_max_sync(full, hi - lo) + 7) / 8;   // of an orbital
            cplx x = cz();
            for (int q0 = 0; q0 < D * steps; q0 += 4) {
                cplx w[4], e[4];
                bool any = false;
#pragma unroll
                for (int z = 0; z < 4; ++z) {
                    const int co = (q0 + z) / steps, c = lo + (lane & 7) + 8 * (q0 + z - co * steps);
                    const int j = s.rowc ? c : f, m = s.rowc ? f : c;
                    w[z] = e[z] = cz();
                    if (co < D && c < hi && histu_has(s, j, m)) {
                        w[z] = v[c * D + co];
                        e[z] = histu_el(*t.p, s, D, j, m, s.rowc ? co : fo, s.rowc ? fo : co);
                    }
                }
#pragma unroll
                for (int z = 0; z < 4; ++z) any = any || (nonzero(w[z]) && nonzero(e[z]));
                if (!__any_sync(full, any)) continue;
#pragma unroll
                for (int z = 0; z < 4; ++z) x = cfma(e[z], histu_conj(s.vec) ? cconj(w[z]) : w[z], x);
            }
#pragma unroll
            for (int b = 4; b > 0; b >>= 1) {
                x.x += __shfl_xor_sync(full, x.x, b);
                x.y += __shfl_xor_sync(full, x.y, b);
            }
            if (mine && (lane & 7) == 0) out[r * D] = x;
        }
    }
}

// one warp's 16 free indices of a task; false when a wait ran out
template <int D>
__device__ __forceinline__ bool task_warp(const HistUTab& tab, const Task& t, unsigned char* sm, uint32_t sbase, int warp, int lane,
                                       int& slot, int& ph) {
    const int g = lane >> 2, tt = lane & 3, f0 = t.f0 + warp * 16;
    const unsigned full = 0xffffffffu;
    int4* acc = (int4*)(sm + SM_INT) + warp * 8 * 2 * 32 + lane;   // [output][lo, hi][32]
    const HistUSet s = t.s;
    auto vexp = [&](int o) { return t.p->vexp[(s.vec * D + o) * t.p->q.vch + t.chunk]; };
    bool bad = false;
#pragma unroll
    for (int o = 0; o < D; ++o) bad = bad || vexp(o) < 0;
    // byte offsets of this lane's free indices (g, g + 8) and contracted ones (2t, 2t+1, 2t+8, 2t+9) in a tile
    constexpr int DD16 = D * D * 16;
    const int row_b = (s.rowc ? NGU_M / D : 16 / D) * DD16 + 16;
    const int rs = s.type == 1 ? 16 : D * 16, cs = s.type == 1 ? D * 16 : 16;   // strides of the row and column orbital
    auto off = [&](bool row, int i) { return row ? (i / D) * row_b + (i % D) * rs : (i / D) * DD16 + (i % D) * cs; };
    const int sw = D > 1 ? g & 1 : 0;   // these lanes take the elements of a pair in the other order (bank conflicts)
    int om[2], ok[4], kx[4];
#pragma unroll
    for (int i = 0; i < 2; ++i) om[i] = off(!s.rowc, warp * 16 + g + 8 * i);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        kx[i] = 2 * tt + ((i ^ sw) & 1) + (i >> 1) * 8;
        ok[i] = off(s.rowc, kx[i]);
    }
    const uint32_t pack_hi = sw ? 0x3276u : 0x7632u, pack_lo = sw ? 0x1054u : 0x5410u;
    int uo[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) uo[i] = SM_U + ((g & 3) >= i ? (g >> 2) * 512 + ((g & 3) - i) * 64 : NGH_DIG_B) + tt * 16;

    double val[D];
    float lo[D][4], hi[D][4];
#pragma unroll
    for (int o = 0; o < D; ++o) {
        val[o] = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c) lo[o][c] = hi[o][c] = 0.f;
        acc[o * 64] = acc[o * 64 + 32] = make_int4(0, 0, 0, 0);
    }
    int E = 0, pend = 0;   // scale; tiles in the FP32 accumulators
    auto flush = [&]() {
#pragma unroll
        for (int o = 0; o < D; ++o) {
            int4 x = acc[o * 64], y = acc[o * 64 + 32];
            x.x += f2i(lo[o][0]); x.y += f2i(lo[o][1]); x.z += f2i(lo[o][2]); x.w += f2i(lo[o][3]);
            y.x += f2i(hi[o][0]); y.y += f2i(hi[o][1]); y.z += f2i(hi[o][2]); y.w += f2i(hi[o][3]);
            acc[o * 64] = x;
            acc[o * 64 + 32] = y;
#pragma unroll
            for (int c = 0; c < 4; ++c) lo[o][c] = hi[o][c] = 0.f;
        }
        pend = 0;
    };
    auto take = [&]() {   // the sums so far, at their scale
#pragma unroll
        for (int o = 0; o < D; ++o) {
            const double sc = bad ? 0.0 : pow2(max(E, 128) - 1022 - 20) * pow2(vexp(o) - 1021 - 20);
            val[o] += digits_value(acc[o * 64], acc[o * 64 + 32], sc);
            acc[o * 64] = acc[o * 64 + 32] = make_int4(0, 0, 0, 0);
        }
    };
#pragma unroll 1
    for (int kt = t.kt0; kt < t.kt1; ++kt) {
        if (!mbar_wait(sbase + SM_BAR + slot * 8, ph)) return false;
        const unsigned char* p = sm + slot * TILE_B;
        const unsigned char* up = sm + slot * 8 * U_B;
        const uint32_t empty = sbase + SM_BAR + (ST + slot) * 8;
        if (++slot == ST) { slot = 0; ph ^= 1; }
        // the warp's elements: free indices f0.., contracted 16 kt..; nothing stored or all of it?
        const int fa = f0 / D, fb = (f0 + 15) / D, ka = kt * 16 / D, kb = (kt * 16 + 15) / D;
        const int ja = s.rowc ? ka : fa, jb = s.rowc ? kb : fb, ma = s.rowc ? fa : ka, mb = s.rowc ? fb : kb;
        if (ja >= s.rows || ma >= s.cols || ma >= histu_mend(s, min(jb, s.rows - 1))) {
            __syncwarp();
            if (lane == 0) mbar_arrive(empty);
            continue;
        }
        uint32_t h[2][4][2], l[2][4][2];   // [free g + 8 fh][contracted][re, im]
#pragma unroll
        for (int fh = 0; fh < 2; ++fh)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint4 x = *(const uint4*)(p + om[fh] + ok[i]);
                l[fh][i][0] = x.x; h[fh][i][0] = x.y; l[fh][i][1] = x.z; h[fh][i][1] = x.w;
            }
        if (jb >= s.rows || mb >= histu_mend(s, ja) || (s.type == 3 && !histu_conv(s, ja, jb, ma, mb))) {   // some do not belong
#pragma unroll
            for (int fh = 0; fh < 2; ++fh)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int f = (f0 + g + 8 * fh) / D, c = (kt * 16 + kx[i]) / D, j = s.rowc ? c : f, m = s.rowc ? f : c;
                    if (!histu_has(s, j, m)) h[fh][i][0] = h[fh][i][1] = 0;
                }
        }
        int sh[2][4][2], neg = 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const uint32_t x = (&h[0][0][0])[i];
            neg |= (&sh[0][0][0])[i] = E - (int)((x + x) >> 21);
        }
        if (E == 0 || __any_sync(full, neg < 0)) {   // first tile, or a larger element: a new scale
            int low = 0;
#pragma unroll
            for (int i = 0; i < 16; ++i) low = min(low, (&sh[0][0][0])[i]);
            const int emax = E + __reduce_max_sync(full, -low);
            bad = bad || emax == 2047;
            const int dE = E == 0 ? max(emax + 1, 128) : emax - E + 3;   // a bit of room, then three: the sums so far are set aside
            if (E != 0) { flush(); take(); }
            E += dE;
#pragma unroll
            for (int i = 0; i < 16; ++i) (&sh[0][0][0])[i] += dE;
        }
        uint32_t P[2][2][2][4], S[2][2][2];   // [free][half][re, im]
#pragma unroll
        for (int fh = 0; fh < 2; ++fh)
#pragma unroll
            for (int kh = 0; kh < 2; ++kh)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t xh[2], xl[2];
#pragma unroll
                    for (int z = 0; z < 2; ++z) {
                        const int i = 2 * kh + z;
                        const uint32_t top = __funnelshift_l(l[fh][i][c], h[fh][i][c], 11) | 0x80000000u;
                        const uint64_t M = shr64(((uint64_t)top << 32) | (l[fh][i][c] << 11), sh[fh][i][c]);
                        xh[z] = (uint32_t)(M >> 32);
                        xl[z] = (uint32_t)M;
                    }
                    P[fh][kh][c][0] = __byte_perm(xh[0], xh[1], pack_hi);
                    P[fh][kh][c][1] = __byte_perm(xh[0], xh[1], pack_lo);
                    P[fh][kh][c][2] = __byte_perm(xl[0], xl[1], pack_hi);
                    P[fh][kh][c][3] = __byte_perm(xl[0], xl[1], pack_lo);
                    S[fh][kh][c] = __byte_perm(h[fh][2 * kh][c], h[fh][2 * kh + 1][c], pack_hi) & 0x80008000u;
                }
        uint32_t d[8][2][2][2];
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                (&d[q][0][0][0])[i] = __byte_perm((&P[0][0][0][0])[i * 4 + (q >> 1)], (&S[0][0][0])[i], (q & 1) ? 0x7250 : 0x7351);
        constexpr int NO = D < 2 ? 1 : 2;   // outputs together: neighbouring products have different accumulators
#pragma unroll
        for (int o0 = 0; o0 < D; o0 += NO)
#pragma unroll
            for (int i = 0; i < 4; ++i) {   // digits (g & 3) - i and (g & 3) + 4 - i of the vector
                uint4 x[NO], y[NO];
#pragma unroll
                for (int o = 0; o < NO; ++o) {
                    const unsigned char* uu = up + (o0 + o) * U_B;
                    x[o] = *(const uint4*)(uu + uo[i]);
                    y[o] = *(const uint4*)(uu + uo[0] + (4 - i) * 64);
                }
                auto first = [&](float(&R)[4], const uint32_t(&e)[2][2][2], const uint4& v) {
                    mma(R, e[0][0][0], e[1][0][0], e[0][0][1], e[1][0][1], v.x, v.y);
                };
                auto second = [&](float(&R)[4], const uint32_t(&e)[2][2][2], const uint4& v) {
                    mma(R, e[0][1][0], e[1][1][0], e[0][1][1], e[1][1][1], v.z, v.w);
                };
#pragma unroll
                for (int o = 0; o < NO; ++o) first(hi[o0 + o], d[i], y[o]);
#pragma unroll
                for (int o = 0; o < NO; ++o) first(lo[o0 + o], d[i], x[o]);
#pragma unroll
                for (int o = 0; o < NO; ++o) second(hi[o0 + o], d[i], y[o]);
#pragma unroll
                for (int o = 0; o < NO; ++o) second(lo[o0 + o], d[i], x[o]);
#pragma unroll
                for (int o = 0; o < NO; ++o) first(hi[o0 + o], d[i + 4], x[o]);
#pragma unroll
                for (int o = 0; o < NO; ++o) second(hi[o0 + o], d[i + 4], x[o]);
            }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty);
        if (++pend == 2) flush();   // 32 contracted elements
    }
    flush();
    take();
    cplx* out = t.p->part + t.p->q.poff[t.set] + ((int64_t)t.chunk * t.p->q.free_[t.set] + f0) * D;
    if (!bad) {
#pragma unroll
        for (int o = 0; o < D; ++o) ((double*)(out + (g + 8 * (tt & 1)) * D + o))[tt >> 1] = val[o];
        if (lane == 0) tab.uexp[((int*)(sm + SM_TASK))[warp] * 8 + warp] = (int)(t.p - tab.probs) << 16 | D << 12 | E;
        return true;
    }
    // a non-finite element or vector: the sums on the FP64 pipe, lane -> (free index, output)
    if (lane == 0) tab.uexp[((int*)(sm + SM_TASK))[warp] * 8 + warp] = 0;
    const cplx* v = t.p->vec + (int64_t)s.vec * D * t.p->q.lenp;
    for (int q = lane; q < 16 * D; q += 32) {
        const int f = (f0 + q / D) / D, fo = (f0 + q / D) % D, o = q % D;
        cplx x = cz();
        for (int c = t.kt0 * 16 / D; c < (t.kt1 * 16 + D - 1) / D; ++c) {
            const int j = s.rowc ? c : f, m = s.rowc ? f : c;
            if (!histu_has(s, j, m)) continue;
            for (int co = 0; co < D; ++co) {
                const cplx w = v[(int64_t)o * t.p->q.lenp + c * D + co];
                x = cfma(histu_el(*t.p, s, D, j, m, s.rowc ? co : fo, s.rowc ? fo : co), histu_conj(s.vec) ? cconj(w) : w, x);
            }
        }
        out[q] = x;
    }
    return true;
}

__global__ void __launch_bounds__(THREADS, 1) k_histu_mma(const __grid_constant__ HistUTab tab) {
    dep_wait();
    extern __shared__ __align__(1024) unsigned char sm[];
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int i = 0; i < ST; ++i) {
            mbar_init(sbase + SM_BAR + i * 8, 1);
            mbar_init(sbase + SM_BAR + (ST + i) * 8, 8);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(sbase + SM_WQ + i * 8, 1);
            mbar_init(sbase + SM_WQ + 16 + i * 8, 8);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < ST * 8 * 4)
        ((uint4*)(sm + SM_U + (threadIdx.x >> 2) * U_B + NGH_DIG_B))[threadIdx.x & 3] = make_uint4(0, 0, 0, 0);
    int* wq = (int*)(sm + SM_WQ + 32);
    __syncthreads();
    // registers of the launch: 12 x 32 x 168; the consumers take 224, the others keep 40
    if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == 8) produce(tab, sbase, wq, lane);
        return;
    }
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    int slot = 0, ph = 0;
    for (int w = 0, wph = 0;;) {
        bool ok = mbar_wait(sbase + SM_WQ + w * 8, wph);
        if (!ok) {
            if (lane == 0) atomicOr(tab.status, NGF_TIMEOUT);
            return;
        }
        const int tk = ((volatile int*)wq)[w];
        __syncwarp();
        if (lane == 0) mbar_arrive(sbase + SM_WQ + 16 + w * 8);
        if (++w == 2) { w = 0; wph ^= 1; }
        if (tk < 0) return;
        const Task t = task_of(tab, tk);
        if (lane == 0) ((int*)(sm + SM_TASK))[warp] = tk;
        switch (t.D) {
            case 1: ok = task_warp<1>(tab, t, sm, sbase, warp, lane, slot, ph); break;
            case 2: ok = task_warp<2>(tab, t, sm, sbase, warp, lane, slot, ph); break;
            case 4: ok = task_warp<4>(tab, t, sm, sbase, warp, lane, slot, ph); break;
            default: ok = task_warp<8>(tab, t, sm, sbase, warp, lane, slot, ph); break;
        }
        if (!ok) {
            if (lane == 0) atomicOr(tab.status, NGF_TIMEOUT);
            return;
        }
    }
}

}  // namespace

cudaError_t histu_launch(const HistUTab& tab, int sms, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_histu_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, SM_BYTES);
    if (e != cudaSuccess) return e;
    dep_launch(k_histu_mma, tab.ntask < sms ? tab.ntask : sms, THREADS, SM_BYTES, s)(tab);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int64_t blocks = (int64_t)tab.ntask * 2 * tab.dmax;
    dep_launch(k_histu_small, (unsigned)(blocks < 16 * sms ? blocks : 16 * sms), 128, 0, s)(tab);
    return cudaGetLastError();
}
