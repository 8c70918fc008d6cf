// sell_long.cuh -- the rows longer than kSeg of single products and batches, in
// kernels of their own that run ahead of the short rows' (sell_spmv_impl.cuh,
// sell_batch.cu).
//
// Work: lwork lists the virtual warps (LongWork).  In a chunk of mostly long
// rows (mode 0) a virtual warp takes one segment of 32 neighbouring rows; in
// a chunk with few long rows (mode 1) it takes 32 consecutive segments of one
// long row after another -- only as many virtual warps as there are segments.
// The chunk holds such a row with a stride of C entries, one useful entry per
// 32-byte sector; its virtual warps therefore have a copy of their entries,
// entry j of lane t at base + j * n + t, n the lanes that have a segment (lval,
// lcol: kSeg entries per segment, less than a quarter of the chunk they come
// from), so that they read like a chunk of n full rows.
// Chunk heights that are not a multiple of 32 go through the units of
// sell_rowdot.cuh instead (lwork is null).
//
// Why a kernel of its own: with both paths in one kernel the long rows' fold
// and loads set the registers of the short rows as well (binary64, one
// vector: 56 against 32, i.e. 32 against 64 warps per SM).  The short rows'
// kernel is launched behind this one as a programmatic dependent: its blocks
// start as soon as every block of this kernel has started, so the two share
// the chip, long rows first, and one thread of it waits for this kernel's end
// before the whole product counts as finished.
//
// Every segment is the chain defined in sell_rowdot.cuh and the partials are
// folded in segment order, so the results are the same bits.
//
// Bounds and measurements (binary64, one vector, block 128, against the long
// rows in the first blocks of the short rows' launch): 10^6 rows of 3 and one
// of 10^6 entries 70 -> 38 us (the row alone 29 us: 8 round trips of loads,
// then chains of 256 and 62 dependent additions at 64 cycles each, the FP64
// pipe's time for a warp); 500,000 lognormal rows unsorted 151 -> 112 us;
// dense 8000^2 147 -> 127 us (FP64 pipe 104 us); 2M lognormal rows sorted
// 133 -> 131 us (gathers).  Tried and slower: a block per 16 segments with
// its entries in shared memory (200,000 sorted rows 26 -> 52 us, dense 402
// us); 16 loads in flight (dense 144 us); prefetches of the packed entries
// (500,000 unsorted rows 132 us).
#pragma once

#include "sell_rowdot.cuh"

namespace sell {

__device__ __forceinline__ void dependents_may_start() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

constexpr int kLongThreads = 128;

// The arrays of a matrix that the long rows need.
struct LongArgs {
    const int32_t *col;
    const int64_t *cs;
    const int32_t *srl, *perm, *lchunk, *lrow;
    const int2 *lunit;
    const LongMeta *lmeta;
    const LongWork *lwork;
    const int32_t *lcol;
    Pattern pt;
    int64_t nwork;  // virtual warps (lwork), or units (lunit) without lwork
    int64_t N;
    int C;
};

// One segment of a long row: long chunk lc, lane l of it, segment s of nseg;
// its entry j is at base + j * stride of val / col, or of lval / lcol.
struct LongSeg {
    int64_t c, r, u0, base;  // chunk, sorted row, the chunk's first partial slot
    int lc, l, s, nseg, L, stride;
    bool valid, packed;
};

__device__ __forceinline__ void finish_segment(const LongArgs &a, LongSeg &g, bool in) {
    g.r = g.c * a.C + g.l;
    g.L = in && g.r < a.N ? a.srl[g.r] : 0;
    g.nseg = (g.L - 1) / kSeg + 1;
    g.valid = g.L > kSeg && g.s < g.nseg;
}

// Lane t of virtual warp w.
__device__ __forceinline__ LongSeg long_segment(const LongArgs &a, int64_t w, int t) {
    LongSeg g;
    const LongWork wk = a.lwork[w];
    g.lc = wk.lc;
    g.c = wk.c;
    g.u0 = wk.u0;
    g.base = wk.base + t;
    bool in = true;
    if (wk.m < 0) {
        const int spc = a.C >> 5;
        g.s = wk.i / spc;
        g.l = (wk.i - g.s * spc) * 32 + t;
        g.stride = a.C;
    } else {
        const int64_t i = (int64_t)wk.i * 32 + t;
        const int64_t k = i / wk.nseg;
        in = k < wk.m;
        g.s = (int)(i - k * wk.nseg);
        g.l = in ? a.lrow[(int64_t)wk.lc * a.C + k] : 0;
        g.stride = (int)min((int64_t)32, (int64_t)wk.m * wk.nseg - (int64_t)wk.i * 32);
    }
    g.packed = wk.m >= 0;
    finish_segment(a, g, in);
    return g;
}

// Unit-thread v (chunk heights that are no multiple of 32).
__device__ __forceinline__ LongSeg unit_segment(const LongArgs &a, int64_t v) {
    LongSeg g;
    const int64_t u = v / a.C;
    const int t = (int)(v - u * a.C);
    if (u >= a.nwork) return LongSeg{};
    const int2 us = a.lunit[u];
    const LongMeta meta = a.lmeta[us.x];
    bool in = true;
    g.lc = us.x;
    g.u0 = u - us.y;
    g.c = a.lchunk[us.x];
    if (meta.mode == 0) {
        g.l = t;
        g.s = us.y;
    } else {
        const int64_t i = (int64_t)us.y * a.C + t;  // beyond 32 bits for rows of more than 2^31 / C segments
        const int64_t k = i / meta.nseg;
        in = k < meta.m;
        g.s = (int)(i - k * meta.nseg);
        g.l = in ? a.lrow[(int64_t)us.x * a.C + k] : 0;
    }
    g.base = a.cs[g.c] + (int64_t)g.s * kSeg * a.C + g.l;
    g.stride = a.C;
    g.packed = false;
    finish_segment(a, g, in);
    return g;
}

__device__ __forceinline__ Plain<double> shfl_acc(const Plain<double> &v, int from) {
    Plain<double> r;
    r.s = __shfl_sync(0xffffffffu, v.s, from);
    return r;
}
__device__ __forceinline__ Dot2 shfl_acc(const Dot2 &v, int from) {
    Dot2 r;
    r.p = __shfl_sync(0xffffffffu, v.p, from);
    r.e = __shfl_sync(0xffffffffu, v.e, from);
    return r;
}

// Folds, for the lanes with `done`, `count` partials each (as fold_partials).
// Either one row after another with the whole warp: lane t adds up column
// t % K, 32 / K partials come with one load of all lanes, a few loads in
// flight.  Or every row in its own lane, all rows at once.  A warp's binary64
// addition takes 64 cycles of the FP64 pipe whatever its lanes do (about twice
// that with the shuffle that brings its operand) and a round trip to L2 the
// time of about kTrip of them, so what counts is the number of additions and
// trips that follow each other.  Measured, before (rows one by one up to
// four, K * n additions each) and after: a row of 10^4 entries in 10^4 short
// ones, eight vectors, binary64 94 -> 45 us, binary32 72 -> 23 us; 1M unsorted
// lognormal rows binary32 at eight vectors 288 -> 249 us; dense 1000^2 the
// same (18.7 us; 21.9 with eight rows of 16 partials one by one).
// All 32 lanes call.
constexpr int kTrip = 10;
template <int K, class PT>
__device__ __forceinline__ void fold_warp(bool done, const PT *part, int64_t base, int64_t stride, int count, int C,
                                          int l, PT (&tot)[K]) {
    const int lane = threadIdx.x & 31;
    unsigned todo = __ballot_sync(0xffffffffu, done);
    const int rows = __popc(todo), most = __reduce_max_sync(0xffffffffu, done ? count : 0);
    const int trips = 1 + (most - 1) / kFoldLoads<K> + (most - 1) % kFoldLoads<K>;  // fold_partials'
    if (rows > 1 && rows * (kTrip + 2 * most) > kTrip * trips + K * most) {
        if (done) fold_partials<K, PT>(part, base, stride, count, C, l, tot);
        __syncwarp();
        return;
    }
    __syncwarp();  // the owner's fence holds for the loads of the other lanes
    constexpr int P = 32 / K, Q = K == 1 ? 8 : 4;  // partials per load, loads in flight (8 at K >= 2: 8 registers more)
    const int e = lane % K;
    for (; todo; todo &= todo - 1) {
        const int owner = __ffs(todo) - 1;
        const int64_t b = __shfl_sync(0xffffffffu, base, owner);
        const int n = __shfl_sync(0xffffffffu, count, owner), ll = __shfl_sync(0xffffffffu, l, owner);
        PT sum;
        for (int i0 = 0; i0 < n; i0 += P * Q) {
            PT p[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int i = i0 + q * P + lane / K;
                if (i < n) p[q] = PT::load_l2(part + ((b + i * stride) * C + ll) * K + e);
            }
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int m = min(P, n - i0 - q * P);
                for (int t = 0; t < m; ++t) {
                    const PT v = shfl_acc(p[q], t * K + e);
                    if (i0 + q * P + t == 0) sum = v;
                    else sum.merge(v);
                }
            }
        }
#pragma unroll
        for (int c = 0; c < K; ++c) {
            const PT v = shfl_acc(sum, c);
            if (lane == owner) tot[c] = v;
        }
    }
}

// Stores the segments' partials and folds the rows (or groups) that they
// complete.  All 32 lanes call; acc counts where g.valid.
template <class XT, int K, class Acc>
__device__ __forceinline__ void long_finish(const LongArgs &a, const LongSeg &g, const Acc (&acc)[K], void *part,
                                            int32_t *cnt, int32_t *cnt2, XT *Y, int64_t ldy, int vec) {
    using PT = typename PartOf<Acc>::T;
    PT *pp = static_cast<PT *>(part);
    const int C = a.C;
    int32_t *ct = cnt + (int64_t)g.lc * C + g.l;
    bool done = false;
    const bool big = g.valid && g.nseg > kSuper;
    if (g.valid) {
#pragma unroll
        for (int q = 0; q < K; ++q) pp[((g.u0 + g.s) * C + g.l) * K + q] = PartOf<Acc>::from(acc[q]);
    }
    const int s0 = (g.s / kSuper) * kSuper, ng = min(kSuper, g.nseg - s0);
    PT tot[K];
    if (__any_sync(0xffffffffu, big)) {
        int32_t *cg = cnt2 + (g.u0 + s0) * C + g.l;
        bool last = false;  // this lane completed its group
        if (big) {
            __threadfence();
            last = atomicAdd(cg, 1) == ng - 1;
            if (last) __threadfence();
        }
        fold_warp<K, PT>(last, pp, g.u0 + s0, 1, ng, C, g.l, tot);
        if (last) {
            *cg = 0;
#pragma unroll
            for (int q = 0; q < K; ++q) pp[((g.u0 + s0) * C + g.l) * K + q] = tot[q];
            __threadfence();
            done = atomicAdd(ct, 1) == (g.nseg + kSuper - 1) / kSuper - 1;
        }
    }
    if (g.valid && !big) {
        __threadfence();
        done = atomicAdd(ct, 1) == g.nseg - 1;
    }
    if (done) __threadfence();
    // rows of up to kSuper segments fold those, the others their groups
    const unsigned bigs = __ballot_sync(0xffffffffu, done && big);
    if (bigs) fold_warp<K, PT>(done && big, pp, g.u0, kSuper, (g.nseg + kSuper - 1) / kSuper, C, g.l, tot);
    if (__any_sync(0xffffffffu, done && !big)) fold_warp<K, PT>(done && !big, pp, g.u0, 1, g.nseg, C, g.l, tot);
    if (done) {
        const int64_t out = a.perm ? (int64_t)a.perm[g.r] : g.r;
#pragma unroll
        for (int q = 0; q < K; ++q)
            if (has_column<K>(q, vec)) Y[out * ldy + q] = static_cast<XT>(tot[q].result());
        *ct = 0;
    }
}

// Unroll and pipelining of a segment's chain.  There are rarely more virtual
// warps than fit on the chip at once, so loads in flight per thread count for
// more than registers: binary32 at four vectors unroll 4 against 2, 1M
// lognormal rows 96 -> 91 us, 300,000 unsorted 68 -> 62 us; at eight 20,000
// rows 24 -> 21 us.  Binary64 is the other way round (FP64 pipe, registers):
// 1M rows at four vectors 113 us against 115 us.
struct LongShape {
    int unroll;
    bool pipe;
};
template <class VT, int K>
constexpr LongShape long_shape() {
    return K == 1 ? LongShape{8, false} : K == 2 ? LongShape{4, false} : sizeof(VT) == 8 ? LongShape{2, true} : LongShape{4, true};
}

// Thread v of a product's long-row work (v / 32 = virtual warp; all 32 lanes
// of a warp call together, with blocks of a multiple of 32 threads).
template <class VT, int K, int U, bool PIPE, class Acc, bool PAT, class LD>
__device__ __forceinline__ void long_rows(const VT *__restrict__ val, const VT *__restrict__ lval, const LongArgs &a,
                                          void *part, int32_t *cnt, int32_t *cnt2,
                                          const typename XType<VT>::T *__restrict__ X, LD ldx,
                                          typename XType<VT>::T *Y, int64_t ldy, int accumulate, int vec, int64_t v) {
    using XT = typename XType<VT>::T;
    LongSeg g;
    if (a.lwork) {
        if (v / 32 >= a.nwork) return;
        g = long_segment(a, v / 32, threadIdx.x & 31);
    } else {
        g = unit_segment(a, v);
    }
    const uint64_t pol = l2_evict_first_policy();
    Acc acc[K];
    if (g.valid) {
        const int64_t out = a.perm ? (int64_t)a.perm[g.r] : g.r;
#pragma unroll
        for (int q = 0; q < K; ++q)
            acc[q].init((g.s == 0 && accumulate && has_column<K>(q, vec)) ? Y[out * ldy + q] : XT(0));
        const int n = min(g.L - g.s * kSeg, kSeg);
        const VT *vp = (g.packed ? lval : val) + g.base;
        bool done = false;
        if constexpr (PAT) {
            if (!g.packed && a.pt.flag[g.r >> 5]) {
                const int64_t cs0 = a.cs[g.c];
                const int32_t *op = a.pt.off + offset_start(cs0, a.pt.cl[g.c], g.l >> 5, g.r >> 5) + g.s * kSeg;
                chain_pattern<VT, XT, K, U, PIPE, 0, Acc>(acc, vp, op, __ldg(a.col + cs0 + g.l), g.stride, n, X, ldx,
                                                          vec, pol);
                done = true;
            }
        }
        if (!done)
            chain<VT, XT, K, U, PIPE, Acc>(acc, vp, (g.packed ? a.lcol : a.col) + g.base, g.stride, 0, n, X, ldx,
                                           vec, pol);
    }
    __syncwarp();
    long_finish<XT, K, Acc>(a, g, acc, part, cnt, cnt2, Y, ldy, vec);
}

template <class VT, int K, int U, bool PIPE, class Acc, bool PAT, class LD>
__global__ void __launch_bounds__(kLongThreads)
k_long(const VT *__restrict__ val, const VT *__restrict__ lval, const LongArgs a, void *part, int32_t *cnt,
       int32_t *cnt2, const typename XType<VT>::T *__restrict__ X, LD ldx, typename XType<VT>::T *Y,
       int64_t ldy, int accumulate, int vec) {
    dependents_may_start();
    long_rows<VT, K, U, PIPE, Acc, PAT>(val, lval, a, part, cnt, cnt2, X, ldx, Y, ldy, accumulate, vec,
                                        blockIdx.x * (int64_t)kLongThreads + threadIdx.x);
}

// The long-row arguments of a handle (with its column patterns or not).
inline LongArgs long_args(const sell_matrix *h, bool pattern) {
    LongArgs a;
    a.col = h->col;
    a.cs = h->cs;
    a.srl = h->srl;
    a.perm = (h->flags & SELL_BUILD_PERMUTE_COLS) ? nullptr : h->perm;
    a.lchunk = h->lchunk;
    a.lrow = h->lrow;
    a.lunit = h->lunit;
    a.lmeta = h->lmeta;
    a.lwork = h->lwork;
    a.lcol = h->lcol;
    a.pt = pattern ? Pattern{h->scol, h->sflag, h->cl} : Pattern{};
    a.nwork = h->lwork ? h->nlwork : h->nunits;
    a.N = h->nrows;
    a.C = h->C;
    return a;
}
// Its threads.
inline int64_t long_threads(const sell_matrix *h) { return h->lwork ? h->nlwork * 32 : h->nunits * h->C; }

}  // namespace sell
