// sell_build.cu -- CRS -> SELL-C-sigma conversion on the GPU (Sec. 3.3-3.4).
//
// Pipeline (one stream, three host synchronisations):
//   k_rowlen                rowLen[i] = rpt[i+1] - rpt[i]; validation of rpt;
//                           max row length and sum of squares (for Eq. "cv")
//   -- sync 1: validation word, max row length --
//   sorting scope sigma     sigma <= 1: identity (no permutation stored)
//                           sigma' = min(sigma, N) <= 4096: k_window_sort, a
//                             bitonic sort in shared memory of whole windows,
//                             several windows per block for small sigma
//                           larger: stable LSD radix sort over the key
//                             (window, maxlen - rowLen), 8-bit digits
//   k_chunk_len             sorted row lengths srl[r], cl[c] = max (Eq. "max")
//   k_chunk_reduce/apply    cs = exclusive prefix sum of C * cl (cl[i] =
//                           (cs[i+1]-cs[i])/C), long chunks, their work units
//   -- sync 2: stored size cs[Nc], long chunks, work units --
//   k_long_lists            the long chunks' work lists
//   k_scatter_tiled         entry j of sorted row r = c*C + l -> cs[c] + j*C + l,
//   (k_scatter)             zero padding (value 0, column 0), value rounding;
//                           validation of col
//   -- sync 3: validation word --
//
// Every sort key is unique (it ends in the row's position), so any correct
// sort gives the stable order: ties in length keep the original row order.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "sell_internal.cuh"

namespace sell {
namespace {

constexpr int kSortKeys = 4096;  // rows per block of the shared-memory sort
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;          // items per thread in the scan
constexpr int kScanTile = kScanThreads * kScanItems;
constexpr int kRadixThreads = 256;
constexpr int kRadixRounds = 8;
constexpr int kRadixTile = kRadixThreads * kRadixRounds;

constexpr int kNopatSlots = 64;  // counters, so that warps rarely meet on one

struct BuildStats {
    unsigned int err;
    int max_rl;
    unsigned long long sumsq;
    unsigned long long nopat[kNopatSlots];  // entries in slices without a column pattern
    unsigned int far;  // slices whose rows begin far apart, of those looked at (k_chunk_len)
};
enum : unsigned int {
    kErrRpt0 = 1u,
    kErrRptOrder = 2u,
    kErrRptEnd = 4u,
    kErrRowLong = 8u,
    kErrCol = 16u,
};

inline int grid_for(int64_t n, int threads, int64_t cap = 1 << 20) {
    int64_t g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    return (int)std::min<int64_t>(g, cap);
}

// ------------------------------------------------------------ row lengths
// Four rows per thread and step, one set of atomics per block: with one set
// per warp of a 2432-block grid, the 58,000 atomics on one cache line took
// most of the kernel's 32 us at 2M rows (24 MB: 3.5 us at 6.8 TB/s).
__global__ void __launch_bounds__(256) k_rowlen(const int64_t *__restrict__ rpt, int64_t N, int64_t nnz,
                                                int32_t *__restrict__ rl, BuildStats *st) {
    __shared__ unsigned int werr[8];
    __shared__ int wmx[8];
    __shared__ unsigned long long wsq[8];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned int err = 0;
    int mx = 0;
    unsigned long long sq = 0;
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 < N; i0 += 4 * stride) {
        int64_t a[4], b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * stride;
            a[q] = i < N ? rpt[i] : 0;
            b[q] = i < N ? rpt[i + 1] : 0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + q * stride;
            if (i >= N) break;
            int64_t len = b[q] - a[q];
            if (i == 0 && a[q] != 0) err |= kErrRpt0;
            if (i == N - 1 && b[q] != nnz) err |= kErrRptEnd;
            if (len < 0) { err |= kErrRptOrder; len = 0; }
            if (len > 0x7FFFFFFF) { err |= kErrRowLong; len = 0; }
            rl[i] = (int32_t)len;
            mx = max(mx, (int)len);
            sq += (unsigned long long)len * (unsigned long long)len;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        err |= __shfl_xor_sync(0xffffffffu, err, o);
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        sq += __shfl_xor_sync(0xffffffffu, sq, o);
    }
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        werr[warp] = err;
        wmx[warp] = mx;
        wsq[warp] = sq;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i) {
            err |= werr[i];
            mx = max(mx, wmx[i]);
            sq += wsq[i];
        }
        if (err) atomicOr(&st->err, err);
        atomicMax(&st->max_rl, mx);
        atomicAdd(&st->sumsq, sq);
    }
}

// ------------------------------------------------- window sort (small sigma)
// One block sorts `wpb` whole windows of W rows (wpb * W <= 4096) with a
// bitonic network over 4096 keys.  Key layout (ascending): window index inside
// the block, max_rl - rowLen (descending length, lbits wide), row position
// inside the block (12 bits, tie-break: original order); KT is 32 bits where
// that fits.  A step of distance j compares keys j apart: up to 32 that stays
// inside the 64 keys that a warp holds in registers (two per lane, exchanged
// by shuffles), so that all stages up to 64 keys are one pass over shared
// memory, and only the 21 wider steps of the network go through it with the
// whole block waiting.  1M rows in windows of 4096 take 30 us, with every
// step in shared memory and 64-bit keys they took 65 us.
// A window length that is a power of two needs no merges across windows: its
// last stage (kmax) sorts every window upwards.
// The steps of distance jmax, jmax / 2 .. 1 of stage k for keys i (a) and
// i + 32 (b), i = 64 * n + lane.
template <class KT>
__device__ __forceinline__ void sort_steps(KT &a, KT &b, int i, int k, int jmax, int kmax) {
    const bool ua = k == kmax || (i & k) == 0, ub = k == kmax || ((i + 32) & k) == 0;
    if (jmax >= 32 && (a > b) == ua) {
        const KT t = a;
        a = b;
        b = t;
    }
    for (int j = min(jmax, 16); j > 0; j >>= 1) {
        const KT pa = __shfl_xor_sync(0xffffffffu, a, j), pb = __shfl_xor_sync(0xffffffffu, b, j);
        const bool low = (i & j) == 0;
        a = (low == ua) == (a > pa) ? pa : a;
        b = (low == ub) == (b > pb) ? pb : b;
    }
}

template <class KT>
__global__ void __launch_bounds__(1024) k_window_sort(const int32_t *__restrict__ rl, int64_t N, int64_t W, int wpb,
                                                      int lbits, int max_rl, int32_t *__restrict__ perm) {
    __shared__ KT key[kSortKeys];
    const int64_t tile = (int64_t)wpb * W;
    const int64_t base = blockIdx.x * tile;
    const int nrow = (int)min(tile, N - base);
    const int kmax = (W & (W - 1)) == 0 ? (int)W : kSortKeys;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto key_of = [&](int i) {
        if (i >= nrow) return (KT)~(KT)0;
        const uint32_t w = (uint32_t)i / (uint32_t)W;
        const KT len = ((KT)(max_rl - rl[base + i]) << 12) | (KT)i;
        return w ? ((KT)w << (12 + lbits)) | len : len;
    };
    for (int i0 = warp * 64; i0 < kSortKeys; i0 += 2048) {
        const int i = i0 + lane;
        KT a = key_of(i), b = key_of(i + 32);
        for (int k = 2; k <= min(64, kmax); k <<= 1) sort_steps(a, b, i, k, k >> 1, kmax);
        key[i] = a;
        key[i + 32] = b;
    }
    for (int k = 128; k <= kmax; k <<= 1) {
        __syncthreads();
        for (int lj = __ffs(k) - 2; lj >= 6; --lj) {
            const int j = 1 << lj;
            for (int t = threadIdx.x; t < kSortKeys / 2; t += 1024) {
                const int lo = ((t >> lj) << (lj + 1)) | (t & (j - 1));
                const bool up = k == kmax || (lo & k) == 0;
                const KT a = key[lo], b = key[lo + j];
                if ((a > b) == up) {
                    key[lo] = b;
                    key[lo + j] = a;
                }
            }
            __syncthreads();
        }
        for (int i0 = warp * 64; i0 < kSortKeys; i0 += 2048) {
            const int i = i0 + lane;
            KT a = key[i], b = key[i + 32];
            sort_steps(a, b, i, k, 32, kmax);
            key[i] = a;
            key[i + 32] = b;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nrow; i += 1024) perm[base + i] = (int32_t)(base + (int64_t)(key[i] & 0xFFF));
}

// --------------------------------------------------- radix sort (large sigma)
// The key of row i: (window, max_rl - rowLen).  The first pass computes it
// from the row lengths (and the row number is the value), so no pass over
// memory writes the initial pairs; KT is 32 bits where the key fits, which
// halves what the later passes move.
template <class KT, bool FIRST>
__device__ __forceinline__ KT radix_key(const KT *__restrict__ key, const int32_t *__restrict__ rl, int64_t i,
                                        uint32_t sigma, int lbits, int max_rl) {
    if constexpr (FIRST) {
        const KT len = (KT)(max_rl - rl[i]);
        const uint32_t w = (uint32_t)i / sigma;
        return w ? ((KT)w << lbits) | len : len;
    } else {
        return key[i];
    }
}

template <class KT, bool FIRST>
__global__ void k_radix_hist(const KT *__restrict__ key, const int32_t *__restrict__ rl, int64_t N, uint32_t sigma,
                             int lbits, int max_rl, int shift, int64_t ntiles, uint32_t *__restrict__ hist) {
    __shared__ uint32_t cnt[256];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t t0 = blockIdx.x * (int64_t)kRadixTile;
#pragma unroll
    for (int r = 0; r < kRadixRounds; ++r) {
        int64_t i = t0 + r * kRadixThreads + threadIdx.x;
        if (i < N) atomicAdd(&cnt[(radix_key<KT, FIRST>(key, rl, i, sigma, lbits, max_rl) >> shift) & 0xFF], 1u);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
}

// Stable scatter of one tile: items are taken in rounds of 256 (thread order
// inside a round, rounds in order); an item's rank is the number of earlier
// items of the tile with the same digit.  All rounds' items are loaded before
// the first is ranked.
template <class KT, bool FIRST>
__global__ void __launch_bounds__(kRadixThreads)
k_radix_scatter(const KT *__restrict__ kin, const int32_t *__restrict__ vin, KT *__restrict__ kout,
                int32_t *__restrict__ vout, const int32_t *__restrict__ rl, int64_t N, uint32_t sigma, int lbits,
                int max_rl, int shift, int64_t ntiles, const int64_t *__restrict__ off) {
    __shared__ int64_t base[256];
    __shared__ uint32_t wcount[kRadixThreads / 32][256];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t t0 = blockIdx.x * (int64_t)kRadixTile;
    KT k[kRadixRounds];
    int32_t v[kRadixRounds];
#pragma unroll
    for (int r = 0; r < kRadixRounds; ++r) {
        const int64_t i = t0 + r * kRadixThreads + tid;
        k[r] = i < N ? radix_key<KT, FIRST>(kin, rl, i, sigma, lbits, max_rl) : (KT)0;
        v[r] = FIRST ? (int32_t)i : (i < N ? vin[i] : 0);
    }
    base[tid] = off[(int64_t)tid * ntiles + blockIdx.x];
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < kRadixRounds; ++r) {
        for (int w = 0; w < kRadixThreads / 32; ++w) wcount[w][tid] = 0;
        __syncthreads();
        const bool valid = t0 + r * kRadixThreads + tid < N;
        const unsigned d = valid ? (unsigned)((k[r] >> shift) & 0xFF) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const unsigned rank = __popc(peers & lt);
        if (valid && rank == 0) wcount[warp][d] = __popc(peers);
        __syncthreads();
        // column tid of the counts: exclusive prefix over the warps
        uint32_t tot = 0;
        for (int w = 0; w < kRadixThreads / 32; ++w) {
            const uint32_t n = wcount[w][tid];
            wcount[w][tid] = tot;
            tot += n;
        }
        __syncthreads();
        if (valid) {
            const int64_t pos = base[d] + wcount[warp][d] + rank;
            kout[pos] = k[r];
            vout[pos] = v[r];
        }
        __syncthreads();
        base[tid] += tot;
    }
}

// -------------------------------------------------------------- prefix scan
// Exclusive scan of int64 sums: out has n + 1 entries with the total in
// out[n].  Two kernels: sums of 4096-item tiles, then every tile scans its
// items and adds the sum of the tiles before it, which its block adds up
// itself -- one launch less than a scan of the tile sums in between (3 us of
// a small build's every scan); only above kScanFlat tiles, where that sum
// would cost more than it saves, the tile sums are scanned first.
constexpr int64_t kScanFlat = 4096;

__device__ __forceinline__ int64_t block_exclusive(int64_t v, int64_t *warp_tot, int64_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        int64_t u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int nw = blockDim.x >> 5;
        int64_t t = lane < nw ? warp_tot[lane] : 0;
        int64_t ti = t;
        for (int o = 1; o < 32; o <<= 1) {
            int64_t u = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += u;
        }
        if (lane < nw) warp_tot[lane] = ti - t;
        if (lane == nw - 1) *total = ti;
    }
    __syncthreads();
    return inc - v + warp_tot[warp];
}

// The sum of bsum[0..n) (tile sums before this block's tile), by the whole block.
__device__ __forceinline__ int64_t tiles_before(const int64_t *__restrict__ bsum, int64_t n, int64_t *wt) {
    int64_t s = 0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += bsum[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) wt[threadIdx.x >> 5] = s;
    __syncthreads();
    s = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += wt[i];
    __syncthreads();
    return s;
}

template <class T>
__global__ void __launch_bounds__(kScanThreads)
k_scan_reduce(const T *__restrict__ in, int64_t n, int64_t *__restrict__ bsum) {
    __shared__ int64_t wt[32];
    __shared__ int64_t tot;
    int64_t i0 = blockIdx.x * (int64_t)kScanTile + threadIdx.x * kScanItems;
    int64_t s = 0;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q)
        if (i0 + q < n) s += (int64_t)in[i0 + q];
    block_exclusive(s, wt, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

// boff: scanned tile sums; bsum: plain tile sums (added up here); neither
// with a single tile.
template <class T>
__global__ void __launch_bounds__(kScanThreads)
k_scan_apply(const T *__restrict__ in, int64_t n, const int64_t *__restrict__ boff,
             const int64_t *__restrict__ bsum, int64_t *__restrict__ out) {
    __shared__ int64_t wt[32];
    __shared__ int64_t tot;
    const int64_t before = boff ? boff[blockIdx.x] : (bsum ? tiles_before(bsum, blockIdx.x, wt) : 0);
    int64_t i0 = blockIdx.x * (int64_t)kScanTile + threadIdx.x * kScanItems;
    int64_t v[kScanItems];
    int64_t s = 0;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) {
        v[q] = (i0 + q < n) ? (int64_t)in[i0 + q] : 0;
        s += v[q];
    }
    int64_t ex = block_exclusive(s, wt, &tot) + before;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) {
        if (i0 + q < n) out[i0 + q] = ex;
        ex += v[q];
    }
    // the tile total (items past n are zero) completes the last tile
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = before + tot;
}

template <class T>
sell_status scan_exclusive(const T *in, int64_t n, int64_t *out, const Allocator &al, cudaStream_t s) {
    if (n == 0) {
        SELL_CUDA_TRY(cudaMemsetAsync(out, 0, sizeof(int64_t), s));
        return SELL_OK;
    }
    int64_t nb = (n + kScanTile - 1) / kScanTile;
    DevBuf bsum, boff;
    if (nb > 1) {
        SELL_TRY(bsum.alloc(al, nb * sizeof(int64_t), s));
        k_scan_reduce<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, bsum.as<int64_t>());
        SELL_CUDA_TRY(cudaGetLastError());
        if (nb > kScanFlat) {
            SELL_TRY(boff.alloc(al, (nb + 1) * sizeof(int64_t), s));
            SELL_TRY(scan_exclusive<int64_t>(bsum.as<int64_t>(), nb, boff.as<int64_t>(), al, s));
        }
    }
    k_scan_apply<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, boff.as<int64_t>(), bsum.as<int64_t>(), out);
    SELL_CUDA_TRY(cudaGetLastError());
    return SELL_OK;
}

// The sums over the chunks in one scan: chunk offsets (C * cl), long chunks
// (cl > kSeg), their segments (ceil(cl / kSeg) each), the virtual warps of
// sell_long.cuh and the packed segments.  nlr[c] = rows of chunk c longer than kSeg.
// The first long-row warp and packed segment of a chunk.
struct WorkBase {
    int64_t nwork, npack;
};

struct ChunkSums {
    int64_t stored, nlong, nunits, nwork, npack;
    __device__ __forceinline__ ChunkSums &operator+=(const ChunkSums &o) {
        stored += o.stored;
        nlong += o.nlong;
        nunits += o.nunits;
        nwork += o.nwork;
        npack += o.npack;
        return *this;
    }
};
// Whether a chunk with m long rows deals their segments out one row after
// another (mode 1 of k_long_lists).
__device__ __forceinline__ bool few_long(int m, int C) { return 8 * (int64_t)m <= C; }

__device__ __forceinline__ ChunkSums sums_of(const int32_t *__restrict__ cl, const int32_t *__restrict__ nlr,
                                             int64_t c, int C) {
    const int32_t w = cl[c];
    if (w <= kSeg) return {(int64_t)C * w, 0, 0, 0, 0};
    const int64_t nseg = (w - 1) / kSeg + 1;  // no overflow near 2^31
    const int m = nlr[c];
    if (C % 32) return {(int64_t)C * w, 1, nseg, 0, 0};
    if (!few_long(m, C)) return {(int64_t)C * w, 1, nseg, nseg * (C / 32), 0};
    return {(int64_t)C * w, 1, nseg, (m * nseg + 31) / 32, m * nseg};
}
__device__ __forceinline__ ChunkSums shfl_up(const ChunkSums &v, int o) {
    return {__shfl_up_sync(0xffffffffu, v.stored, o), __shfl_up_sync(0xffffffffu, v.nlong, o),
            __shfl_up_sync(0xffffffffu, v.nunits, o), __shfl_up_sync(0xffffffffu, v.nwork, o),
            __shfl_up_sync(0xffffffffu, v.npack, o)};
}
// Inclusive scan over the block (1024 threads); *tot = the block's total.
__device__ __forceinline__ ChunkSums block_inclusive(ChunkSums v, ChunkSums *wt) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const ChunkSums u = shfl_up(v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) wt[warp] = v;
    __syncthreads();
    if (warp == 0) {
        ChunkSums t = wt[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const ChunkSums u = shfl_up(t, o);
            if (lane >= o) t += u;
        }
        __syncwarp();
        wt[lane] = t;
    }
    __syncthreads();
    if (warp > 0) v += wt[warp - 1];
    return v;
}

// Sums of tiles of `per` chunks (a multiple of 1024), one tile per block.
__global__ void __launch_bounds__(kScanThreads)
k_chunk_reduce(const int32_t *__restrict__ cl, const int32_t *__restrict__ nlr, int64_t Nc, int64_t per, int C,
               ChunkSums *__restrict__ tile) {
    __shared__ ChunkSums wt[32];
    const int64_t c0 = blockIdx.x * per, c1 = min(Nc, c0 + per);
    ChunkSums v = {0, 0, 0, 0, 0};
    for (int64_t c = c0 + threadIdx.x; c < c1; c += kScanThreads) v += sums_of(cl, nlr, c, C);
    v = block_inclusive(v, wt);
    if (threadIdx.x == kScanThreads - 1) tile[blockIdx.x] = v;
}

// cs, and for the long chunks their index, first unit and first virtual warp
// (and first packed one) in lpos/ubase/wbase; the totals go to cs[Nc] and *total.  tile: the tile sums.
// dot_count (may be null): sell_spmv_dot's count of finished blocks, zero between products.
__global__ void __launch_bounds__(kScanThreads)
k_chunk_apply(const int32_t *__restrict__ cl, const int32_t *__restrict__ nlr, int64_t Nc, int64_t per, int C,
              const ChunkSums *__restrict__ tile,
              int64_t *__restrict__ cs, int64_t *__restrict__ lpos, int64_t *__restrict__ ubase,
              WorkBase *__restrict__ wbase, ChunkSums *__restrict__ total, int64_t *__restrict__ dot_count) {
    __shared__ ChunkSums wt[32];
    __shared__ ChunkSums before;
    ChunkSums s = {0, 0, 0, 0, 0};
    for (int64_t i = threadIdx.x; i < blockIdx.x; i += kScanThreads) s += tile[i];
    s = block_inclusive(s, wt);
    if (threadIdx.x == kScanThreads - 1) before = s;
    __syncthreads();
    const int64_t c1 = min(Nc, (blockIdx.x + 1) * per);
    for (int64_t c0 = blockIdx.x * per; c0 < c1; c0 += kScanThreads) {
        const int64_t c = c0 + threadIdx.x;
        const ChunkSums own = c < c1 ? sums_of(cl, nlr, c, C) : ChunkSums{0, 0, 0, 0, 0};
        ChunkSums v = block_inclusive(own, wt);
        v += before;
        if (c < c1) {
            cs[c] = v.stored - own.stored;
            lpos[c] = v.nlong - own.nlong;
            ubase[c] = v.nunits - own.nunits;
            wbase[c] = WorkBase{v.nwork - own.nwork, v.npack - own.npack};
            if (c == Nc - 1) {
                cs[Nc] = v.stored;
                *total = v;
                if (dot_count) *dot_count = 0;
            }
        }
        __syncthreads();
        if (threadIdx.x == kScanThreads - 1) before = v;
        __syncthreads();
    }
}

// ------------------------------------------------------------- chunk lengths
// srl, cl, and src[r] = where sorted row r's entries begin in the CRS arrays:
// the scatter then waits for one load instead of a chain of three (length,
// perm, rpt) before a row's entries.
// Every near_step-th slice (32 sorted rows; 0: none) also says whether its rows
// begin kNear columns or more apart (st->far).
constexpr int kNear = 4096;        // rows of X of up to 32 bytes that L1 holds
constexpr int kNearSlices = 1024;  // slices looked at, about
__global__ void k_chunk_len(const int32_t *__restrict__ rl, const int32_t *__restrict__ perm,
                            const int64_t *__restrict__ rpt, int64_t N, int64_t Np, int C, int32_t *__restrict__ srl,
                            int64_t *__restrict__ src, int32_t *__restrict__ cl, int32_t *__restrict__ nlr,
                            int32_t *__restrict__ inv, const int32_t *__restrict__ col_in, int64_t near_step,
                            BuildStats *st) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool warp_chunks = (C % 32) == 0;
    // the loop trip count is uniform across a warp because Np is a multiple of
    // C and the grid stride is a multiple of 32
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r - (threadIdx.x & 31) < Np;
         r += stride) {
        bool live = r < Np;
        int32_t len = 0;
        if (live && r < N) {
            int64_t old = perm ? perm[r] : r;
            len = rl[old];
            if (inv) inv[old] = (int32_t)r;
        }
        if (live) {
            srl[r] = len;
            if (r < N) src[r] = rpt[perm ? perm[r] : r];
        }
        if (near_step && (r >> 5) % near_step == 0) {
            const int32_t first = len > 0 ? col_in[src[r]] : 0;
            const int32_t lo = __reduce_min_sync(0xffffffffu, len > 0 ? first : 0x7FFFFFFF);
            const int32_t hi = __reduce_max_sync(0xffffffffu, len > 0 ? first : 0);
            if ((threadIdx.x & 31) == 0 && (int64_t)hi - lo >= kNear) atomicAdd(&st->far, 1u);
        }
        if (warp_chunks) {
            int32_t m = len;
            for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
            const int nl = __popc(__ballot_sync(0xffffffffu, len > kSeg));
            if (live && (threadIdx.x & 31) == 0 && m > 0) {
                atomicMax(&cl[r / C], m);
                if (nl) atomicAdd(&nlr[r / C], nl);
            }
        } else if (live && len > 0) {
            atomicMax(&cl[r / C], len);
            if (len > kSeg) atomicAdd(&nlr[r / C], 1);
        }
    }
}

// ---------------------------------------------------------- long-row chunks
// The long chunks (cl > kSeg), one warp per chunk: lchunk[i] = the i-th
// long chunk; its ceil(cl / kSeg) work units are lunit[ubase + s] = {i, s};
// lrow[i*C + k] = the lane of its k-th row longer than kSeg (lane order),
// lmeta[i] = {m rows, mode, units of the chunk}.  Mode 0: unit thread t
// takes lane t (its row's segment); mode 1, for chunks whose long rows are
// few (8 m <= C): the chunk's unit threads take consecutive segments of one
// long row after another, so a warp runs 32 segments of a long row instead of
// one segment of each of 32 mostly short rows.  Either way each segment is
// the same chain and lands in the same partial slot (unit of the segment,
// lane of the row), so the results do not depend on the mode.
__global__ void __launch_bounds__(256)
k_long_lists(const int32_t *__restrict__ cl, const int32_t *__restrict__ srl, const int64_t *__restrict__ lpos,
             const int64_t *__restrict__ ubase, const WorkBase *__restrict__ wbase, const int64_t *__restrict__ cs, int64_t Nc, int64_t N, int C,
             int32_t *__restrict__ lchunk, int2 *__restrict__ lunit, int32_t *__restrict__ lrow,
             LongMeta *__restrict__ lmeta, LongWork *__restrict__ lwork) {
    const int lane = threadIdx.x & 31;
    const int64_t c = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    const int32_t width = c < Nc ? cl[c] : 0;
    if (width <= kSeg) return;
    const int64_t i = lpos[c], u = ubase[c];
    const int nseg = (width - 1) / kSeg + 1;
    for (int sg = lane; sg < nseg; sg += 32) lunit[u + sg] = make_int2((int)i, sg);
    int m = 0;
    for (int l0 = 0; l0 < C; l0 += 32) {
        const int64_t r = c * C + l0 + lane;
        const bool lg = l0 + lane < C && r < N && srl[r] > kSeg;
        const unsigned hit = __ballot_sync(0xffffffffu, lg);
        if (lg) lrow[i * C + m + __popc(hit & ((1u << lane) - 1u))] = l0 + lane;
        m += __popc(hit);
    }
    const bool few = few_long(m, C);
    if (lwork) {
        const int64_t n = few ? ((int64_t)m * nseg + 31) / 32 : (int64_t)nseg * (C / 32);
        const WorkBase wb = wbase[c];
        for (int64_t k = lane; k < n; k += 32) {
            LongWork wk;
            wk.lc = (int32_t)i;
            wk.c = (int32_t)c;
            wk.nseg = nseg;
            wk.m = few ? m : -1;
            const int sl = (int)(k % (C / 32)), sg = (int)(k / (C / 32));
            wk.base = few ? (wb.npack + k * 32) * kSeg : cs[c] + (int64_t)sg * kSeg * C + sl * 32;
            wk.i = (int32_t)k;
            wk.u0 = (int32_t)u;
            lwork[wb.nwork + k] = wk;
        }
    }
    if (lane == 0) {
        lchunk[i] = (int32_t)c;
        lmeta[i] = LongMeta{m, few ? 1 : 0, nseg};
    }
}

// ------------------------------------------------- bulk-staged SpMV plan
// bsc[c] = the longest row of at most kSeg entries in chunk c, -1 if the
// chunk has no such row (the columns of chunk c that the bulk-staged SpMV
// copies), and its work weight bw[c] = bsc[c] + 1.  One warp per chunk.
__global__ void k_bulk_cols(const int32_t *__restrict__ srl, int64_t N, int64_t Nc, int C,
                            int32_t *__restrict__ bsc, int32_t *__restrict__ bw) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t c = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); c < Nc; c += nw) {
        int m = -1;
        for (int l = lane; l < C; l += 32) {
            const int len = srl[c * C + l];
            if (c * C + l < N && len <= kSeg) m = max(m, len);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) {
            bsc[c] = m;
            bw[c] = m + 1;
        }
    }
}

// wsplit[w] = first chunk c with bss[c] >= w * total / nw (bss = exclusive
// scan of the weights bw, bss[Nc] = total), wsplit[nw] = Nc: warp w stages
// chunks [wsplit[w], wsplit[w+1]), about total / nw weight.
__global__ void k_bulk_split(const int64_t *__restrict__ bss, int64_t Nc, int64_t nw, int32_t *__restrict__ wsplit) {
    const int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (w > nw) return;
    if (w == nw) {
        wsplit[w] = (int32_t)Nc;
        return;
    }
    const int64_t total = bss[Nc];
    const int64_t target = total * w / nw;  // total <= 64 * Nc < 2^37, w <= nw < 2^20
    int64_t lo = 0, hi = Nc;  // first index in [0, Nc] with bss >= target
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (bss[mid] < target) lo = mid + 1;
        else hi = mid;
    }
    wsplit[w] = (int32_t)lo;
}

// ------------------------------------------------------------------ scatter
template <class TI, class TO> __device__ __forceinline__ TO cvt(TI v);
template <> __device__ __forceinline__ double cvt<double, double>(double v) { return v; }
template <> __device__ __forceinline__ float cvt<double, float>(double v) { return __double2float_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat16 cvt<double, __nv_bfloat16>(double v) {
    return __double2bfloat16(v);
}
template <> __device__ __forceinline__ double cvt<float, double>(float v) { return (double)v; }
template <> __device__ __forceinline__ float cvt<float, float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 cvt<float, __nv_bfloat16>(float v) {
    return __float2bfloat16_rn(v);
}
template <class TO> __device__ __forceinline__ TO zero_of();
template <> __device__ __forceinline__ double zero_of<double>() { return 0.0; }
template <> __device__ __forceinline__ float zero_of<float>() { return 0.0f; }
template <> __device__ __forceinline__ __nv_bfloat16 zero_of<__nv_bfloat16>() {
    return __ushort_as_bfloat16((unsigned short)0);
}

// One thread per sorted row; the C threads of a chunk write one stored column
// (C consecutive elements) per step j.  Chunk heights that are not a multiple
// of 32 only: there a warp's rows span several chunks.
template <class TI, class TO>
__global__ void k_scatter(const int64_t *__restrict__ src_of, const int32_t *__restrict__ col_in,
                          const TI *__restrict__ val_in, const int32_t *__restrict__ inv, const int32_t *__restrict__ srl,
                          const int32_t *__restrict__ cl, const int64_t *__restrict__ cs, int64_t N,
                          int64_t Np, int C, int64_t ncols, TO *__restrict__ val, int32_t *__restrict__ col,
                          BuildStats *st) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < Np; r += stride) {
        int64_t c = r / C;
        int l = (int)(r - c * C);
        int32_t width = cl[c];
        int32_t len = srl[r];
        int64_t src = 0;
        if (r < N) src = src_of[r];
        int64_t pos = cs[c] + l;
        for (int32_t j = 0; j < width; ++j, pos += C) {
            if (j < len) {
                int32_t cidx = col_in[src + j];
                const bool out = cidx < 0 || (int64_t)cidx >= ncols;
                bad |= out;
                val[pos] = cvt<TI, TO>(val_in[src + j]);
                col[pos] = inv && !out ? inv[cidx] : cidx;
            } else {
                val[pos] = zero_of<TO>();
                col[pos] = 0;
            }
        }
    }
    if (bad) atomicOr(&st->err, kErrCol);
}

// Chunk heights of a multiple of 32: one warp per slice (32 consecutive sorted
// rows) and kSeg stored columns, kTileCols of them at a time (and one per
// virtual warp with packed entries, sell_long.cuh).  The warp reads
// the entries row by row -- 16 consecutive entries of two rows per load (4 or
// 8 of more rows where the rows are short), so a row's bytes are read once and
// in whole sectors -- into a shared tile, and writes the tile column by column
// (32 consecutive elements).  The first Np /
// 32 warps take each slice's first kSeg columns, the others the long chunks'
// further segments (lunit), so one very long row does not hold a single warp
// for its whole length.
// Bound: HBM (CRS read once, the format written once: 770 MB and 113 us at
// 6.8 TB/s for 2M lognormal rows in binary64).  The thread-per-row form above
// took 648 us there (two dependent uncoalesced loads in flight per thread),
// this one 235 us: the rows' pieces begin and end inside sectors (1.46 times
// the bytes move) and the warp waits for each batch of loads.  Loads in
// flight: 8 per lane for 8-byte values (235 us; 4: 283 us), 4 for the others
// (1M banded rows to binary32 80 us; 8: 94 us); a branch around each load
// instead of a predicate cost up to 60 % more.
//
// On the way the warp finds out whether its slice has one column pattern: the
// entry j of every row lies at (the row's first column) + off[j], with off[j]
// the same for all rows that have an entry j.  Rows of structured grids away
// from their boundary and of dense blocks do; rows of fewer than kPatternRow
// entries have next to no columns to save and are read as they are (1M rows of
// one entry, binary32 at eight vectors 12.3 us, with offsets 16.3; of three 18.6
// and 18.0).  off[j] goes to scol (at
// offset_start), and sflag[slice] is cleared for slices without a pattern; their
// entries are counted in st->nopat.
constexpr int kTileCols = 16;
constexpr int kPatternRow = 3;

// A read-only load under a predicate, zero otherwise, with no branch around
// it: a batch of them is in flight together.
__device__ __forceinline__ double ld_if(const double *p, bool on) {
    double v;
    asm("{\n .reg .pred q;\n setp.ne.s32 q, %2, 0;\n mov.f64 %0, 0d0000000000000000;\n @q ld.global.nc.f64 %0, [%1];\n}"
        : "=d"(v) : "l"(p), "r"((int)on));
    return v;
}
__device__ __forceinline__ float ld_if(const float *p, bool on) {
    float v;
    asm("{\n .reg .pred q;\n setp.ne.s32 q, %2, 0;\n mov.f32 %0, 0f00000000;\n @q ld.global.nc.f32 %0, [%1];\n}"
        : "=f"(v) : "l"(p), "r"((int)on));
    return v;
}
__device__ __forceinline__ int32_t ld_if(const int32_t *p, bool on) {
    int32_t v;
    asm("{\n .reg .pred q;\n setp.ne.s32 q, %2, 0;\n mov.s32 %0, 0;\n @q ld.global.nc.s32 %0, [%1];\n}"
        : "=r"(v) : "l"(p), "r"((int)on));
    return v;
}
constexpr int kScatterWarps = 4;

template <class TI, class TO>
__global__ void __launch_bounds__(kScatterWarps * 32)
k_scatter_tiled(const int64_t *__restrict__ src_of, const int32_t *__restrict__ col_in,
                const TI *__restrict__ val_in, const int32_t *__restrict__ inv, const int32_t *__restrict__ srl,
                const int32_t *__restrict__ cl, const int64_t *__restrict__ cs, const int32_t *__restrict__ lchunk,
                const int2 *__restrict__ lunit, const int32_t *__restrict__ lrow, const LongWork *__restrict__ lwork,
                int64_t nunits, int64_t nlwork, int64_t N, int64_t nslices, int C, int64_t ncols,
                TO *__restrict__ val, int32_t *__restrict__ col, TO *__restrict__ lval, int32_t *__restrict__ lcol,
                int32_t *__restrict__ scol, int32_t *__restrict__ sflag, BuildStats *st) {
    // row pitches that keep the column-wise writes of a half-warp off each
    // other's banks
    __shared__ TO tval[kScatterWarps][kTileCols][sizeof(TO) == 8 ? 33 : 34];
    __shared__ int32_t tcol[kScatterWarps][kTileCols][34];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t w = blockIdx.x * (int64_t)kScatterWarps + warp;
    const uint32_t spc = (uint32_t)C / 32;  // slices per chunk
    const int64_t npieces = nslices + nunits * spc;
    int64_t slice = 0, src = 0, at, ostart = 0;  // at: where column j0 of the piece begins
    int seg = 0, len, j0 = 0, j1 = kSeg, stride = 32;
    const bool pack = w >= npieces;
    if (!pack) {
        int64_t c;
        uint32_t sl;
        if (w < nslices) {
            c = (uint32_t)w / spc;
            sl = (uint32_t)w % spc;
        } else {
            const int64_t i = w - nslices;
            const int2 us = lunit[i / spc];
            seg = us.y;
            if (seg == 0) return;  // the slice's own warp has the first segment
            sl = (uint32_t)(i % spc);
            c = lchunk[us.x];
        }
        slice = c * spc + sl;
        const int64_t r = slice * 32 + lane, cs0 = cs[c];
        const int width = cl[c];
        len = r < N ? srl[r] : 0;
        src = r < N ? src_of[r] : 0;
        j0 = seg * kSeg;
        j1 = min(width, j0 + kSeg);
        stride = C;
        at = cs0 + (int64_t)j0 * C + sl * 32;
        ostart = offset_start(cs0, width, (int)sl, slice);
    } else {  // a virtual warp of a chunk with few long rows: lane t's segment as a row of its own
        if (w - npieces >= nlwork) return;
        const LongWork wk = lwork[w - npieces];
        if (wk.m < 0) return;
        const int64_t i = (int64_t)wk.i * 32 + lane, k = i / wk.nseg;
        stride = (int)min((int64_t)32, (int64_t)wk.m * wk.nseg - i + lane);
        len = 0;
        if (k < wk.m) {
            const int64_t r = (int64_t)wk.c * C + lrow[(int64_t)wk.lc * C + k];
            const int s0 = (int)(i - k * wk.nseg) * kSeg;
            len = max(0, min(srl[r] - s0, kSeg));
            src = src_of[r] + s0;
        }
        at = wk.base;
        val = lval;
        col = lcol;
    }
    // the row of the tile that this lane writes: the last one again where there
    // are fewer than 32 (no branch around the writes: with one the build of 2M
    // lognormal rows takes 107 us more)
    const int row = min(lane, stride - 1);
    const int wmax = __reduce_max_sync(0xffffffffu, len);
    bool bad = false;
    auto mapped = [&](int32_t cidx) {
        const bool out = cidx < 0 || (int64_t)cidx >= ncols;
        bad |= out;
        return inv && !out ? inv[cidx] : cidx;
    };
    const int lref = __ffs(__ballot_sync(0xffffffffu, len == wmax)) - 1;
    int32_t first = seg > 0 && len > 0 ? mapped(col_in[src]) : 0;  // segment 0 has it in its first tile
    int32_t fref = __shfl_sync(0xffffffffu, first, lref);
    bool same = true;
    auto load_tile = [&](auto lanes_log2, int jt) {
        constexpr int LG = decltype(lanes_log2)::value;
        constexpr int B = sizeof(TO) == 8 ? 8 : 4;  // loads in flight per lane and array, at most 1 << LG
        constexpr int BB = B < (1 << LG) ? B : (1 << LG);
        const int jj = lane & ((1 << LG) - 1);
#pragma unroll 1
        for (int it = 0; it < (1 << LG); it += BB) {
            TI v[BB];
            int32_t ci[BB];
            bool in[BB];
#pragma unroll
            for (int b = 0; b < BB; ++b) {
                const int l = ((it + b) << (5 - LG)) + (lane >> LG);
                const int n = __shfl_sync(0xffffffffu, len, l);
                const int64_t p = __shfl_sync(0xffffffffu, src, l) + jt + jj;
                in[b] = jt + jj < n;
                v[b] = ld_if(val_in + p, in[b]);
                ci[b] = ld_if(col_in + p, in[b]);
            }
#pragma unroll
            for (int b = 0; b < BB; ++b) {
                const int l = ((it + b) << (5 - LG)) + (lane >> LG);
                tval[warp][jj][l] = cvt<TI, TO>(v[b]);  // zero stays zero
                tcol[warp][jj][l] = in[b] ? mapped(ci[b]) : 0;
            }
        }
    };
    for (int jt = j0; jt < j1; jt += kTileCols) {
        if (jt < wmax) {
            // 16 lanes per row, fewer where the rest of the rows is short
            const int rest = wmax - jt;
            if (rest > 8) load_tile(std::integral_constant<int, 4>(), jt);
            else if (rest > 4) load_tile(std::integral_constant<int, 3>(), jt);
            else load_tile(std::integral_constant<int, 2>(), jt);
            __syncwarp();
            if (jt == 0) {
                first = tcol[warp][0][lane];
                fref = __shfl_sync(0xffffffffu, first, lref);
            }
        }
        const int nj = min(kTileCols, j1 - jt);
        int32_t myoff = 0;
        int64_t pos = at + (int64_t)(jt - j0) * stride + row;
        for (int q = 0; q < nj; ++q, pos += stride) {
            if (jt + q < wmax) {
                const int32_t cc = tcol[warp][q][row];
                val[pos] = tval[warp][q][row];
                col[pos] = cc;
                const int32_t off = __shfl_sync(0xffffffffu, cc, lref) - fref;
                same &= jt + q >= len || cc - first == off;
                if (lane == q) myoff = off;
            } else {  // columns that only other slices of the chunk reach
                val[pos] = zero_of<TO>();
                col[pos] = 0;
            }
        }
        if (lane < nj && !pack) scol[ostart + jt + lane] = myoff;
        __syncwarp();
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&st->err, kErrCol);
    if (!pack && (wmax < kPatternRow || !__all_sync(0xffffffffu, same))) {
        unsigned long long n = len;  // the whole slice's, by the first of its pieces to come here
        for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
        if (lane == 0 && atomicExch(&sflag[slice], 0) != 0 && n) atomicAdd(&st->nopat[w % kNopatSlots], n);
    }
}

// Arrays of the format under construction that the scatter reads or writes.
struct ScatterArgs {
    const int64_t *src;
    const int32_t *col_in;
    const void *val_in;
    const int32_t *inv, *srl, *cl;
    const int64_t *cs;
    const int32_t *lchunk;
    const int2 *lunit;
    const int32_t *lrow;
    const LongWork *lwork;
    int64_t nunits, nlwork, N, Np, ncols;
    int C;
    void *val, *lval;
    int32_t *lcol;
    int32_t *col, *scol, *sflag;
    BuildStats *st;
};

template <class TI, class TO>
sell_status run_scatter(const ScatterArgs &a, cudaStream_t s) {
    const TI *vi = static_cast<const TI *>(a.val_in);
    TO *vo = static_cast<TO *>(a.val);
    if (a.C % 32 == 0) {
        const int64_t items = a.Np / 32 + a.nunits * (a.C / 32) + (a.lval ? a.nlwork : 0);
        k_scatter_tiled<TI, TO><<<(unsigned)((items + kScatterWarps - 1) / kScatterWarps), kScatterWarps * 32, 0, s>>>(
            a.src, a.col_in, vi, a.inv, a.srl, a.cl, a.cs, a.lchunk, a.lunit, a.lrow, a.lwork,
            a.nunits, a.nlwork, a.N, a.Np / 32, a.C, a.ncols, vo, a.col, static_cast<TO *>(a.lval), a.lcol, a.scol,
            a.sflag, a.st);
    } else {
        k_scatter<TI, TO><<<grid_for(a.Np, 256), 256, 0, s>>>(a.src, a.col_in, vi, a.inv, a.srl, a.cl, a.cs,
                                                              a.N, a.Np, a.C, a.ncols, vo, a.col, a.st);
    }
    SELL_CUDA_TRY(cudaGetLastError());
    return SELL_OK;
}

template <class TI>
sell_status launch_scatter(const ScatterArgs &a, int store, cudaStream_t s) {
    switch (store) {
        case SELL_F64: return run_scatter<TI, double>(a, s);
        case SELL_F32: return run_scatter<TI, float>(a, s);
        default: return run_scatter<TI, __nv_bfloat16>(a, s);
    }
}

int bits_for(unsigned long long v) {  // bits needed to hold 0..v
    int b = 0;
    while (b < 64 && (v >> b) != 0) ++b;
    return b;
}

// LSD radix sort of the rows by (window, max_rl - rowLen), 8 bits a pass.
template <class KT>
sell_status radix_sort(const int32_t *rl, int64_t N, int64_t sigma, int lbits, int bits, int max_rl, int32_t *perm,
                       const Allocator &al, cudaStream_t s) {
    const int passes = (bits + 7) / 8;
    const int64_t ntiles = (N + kRadixTile - 1) / kRadixTile;
    const uint32_t sg = (uint32_t)std::min<int64_t>(sigma, 0x7FFFFFFF);  // rows are numbered below 2^31
    DevBuf k0, k1, v1, hist, off;
    SELL_TRY(k0.alloc(al, N * sizeof(KT), s));
    SELL_TRY(k1.alloc(al, N * sizeof(KT), s));
    SELL_TRY(v1.alloc(al, N * sizeof(int32_t), s));
    SELL_TRY(hist.alloc(al, 256 * ntiles * sizeof(uint32_t), s));
    SELL_TRY(off.alloc(al, (256 * ntiles + 1) * sizeof(int64_t), s));
    KT *ka = k0.as<KT>(), *kb = k1.as<KT>();
    // the values ping-pong between perm and v1 and end in perm
    int32_t *va = (passes % 2 == 0) ? perm : v1.as<int32_t>();
    int32_t *vb = (passes % 2 == 0) ? v1.as<int32_t>() : perm;
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * p;
        const unsigned nt = (unsigned)ntiles;
        uint32_t *hp = hist.as<uint32_t>();
        if (p == 0) k_radix_hist<KT, true><<<nt, kRadixThreads, 0, s>>>(ka, rl, N, sg, lbits, max_rl, shift, ntiles, hp);
        else k_radix_hist<KT, false><<<nt, kRadixThreads, 0, s>>>(ka, rl, N, sg, lbits, max_rl, shift, ntiles, hp);
        SELL_CUDA_TRY(cudaGetLastError());
        SELL_TRY(scan_exclusive<uint32_t>(hp, 256 * ntiles, off.as<int64_t>(), al, s));
        const int64_t *op = off.as<int64_t>();
        if (p == 0)
            k_radix_scatter<KT, true><<<nt, kRadixThreads, 0, s>>>(ka, va, kb, vb, rl, N, sg, lbits, max_rl, shift,
                                                                   ntiles, op);
        else
            k_radix_scatter<KT, false><<<nt, kRadixThreads, 0, s>>>(ka, va, kb, vb, rl, N, sg, lbits, max_rl, shift,
                                                                    ntiles, op);
        SELL_CUDA_TRY(cudaGetLastError());
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    // after the last swap `va` holds the result and is `perm` by construction
    return SELL_OK;
}

sell_status sort_windows(const int32_t *rl, int64_t N, int64_t sigma, int max_rl, int32_t *perm,
                         const Allocator &al, cudaStream_t s) {
    const int64_t W = std::min<int64_t>(sigma, N);
    if (W <= kSortKeys) {
        const int wpb = (int)std::max<int64_t>(1, kSortKeys / W);
        const int64_t tile = wpb * W;
        const unsigned nblk = (unsigned)((N + tile - 1) / tile);
        const int lb = bits_for((unsigned long long)max_rl), wb = bits_for((unsigned long long)(wpb - 1));
        // (below 32 bits, so that no key is the one of the places past the rows)
        if (12 + lb + wb < 32) k_window_sort<uint32_t><<<nblk, 1024, 0, s>>>(rl, N, W, wpb, lb, max_rl, perm);
        else k_window_sort<unsigned long long><<<nblk, 1024, 0, s>>>(rl, N, W, wpb, lb, max_rl, perm);
        SELL_CUDA_TRY(cudaGetLastError());
        return SELL_OK;
    }
    // LSD radix sort on (window, max_rl - rowLen), stable, values = row ids
    int64_t nwin = (N + sigma - 1) / sigma;
    int lbits = std::max(1, bits_for((unsigned long long)max_rl));
    int wbits = bits_for((unsigned long long)(nwin - 1));
    int total = lbits + wbits;
    if (total > 64) return fail(SELL_EUNSUPPORTED, "sort key wider than 64 bits");
    if (total <= 32) return radix_sort<uint32_t>(rl, N, sigma, lbits, total, max_rl, perm, al, s);
    return radix_sort<unsigned long long>(rl, N, sigma, lbits, total, max_rl, perm, al, s);
}

sell_status validate(const sell_csr *A, const sell_opts *o) {
    if (!A || !o) return fail(SELL_EINVAL, "sell_build: NULL matrix or options");
    if (o->C < 1) return fail(SELL_EINVAL, "sell_build: C must be >= 1");
    if (o->sigma < 1) return fail(SELL_EINVAL, "sell_build: sigma must be >= 1");
    if (o->store_type != SELL_F64 && o->store_type != SELL_F32 && o->store_type != SELL_BF16)
        return fail(SELL_EINVAL, "sell_build: unknown store_type");
    if (o->reserved != 0) return fail(SELL_EINVAL, "sell_build: reserved must be 0");
    if (o->flags & ~SELL_BUILD_PERMUTE_COLS) return fail(SELL_EINVAL, "sell_build: unknown flags");
    if (A->nrows < 0 || A->ncols < 0 || A->nnz < 0)
        return fail(SELL_EINVAL, "sell_build: negative size");
    if (A->nrows > 0x7FFFFFFFll || A->ncols > 0x7FFFFFFFll)
        return fail(SELL_EINVAL, "sell_build: nrows and ncols must be below 2^31");
    if (A->val_type != SELL_F64 && A->val_type != SELL_F32)
        return fail(SELL_EINVAL, "sell_build: val_type must be SELL_F64 or SELL_F32");
    if (!A->rpt) return fail(SELL_EINVAL, "sell_build: NULL rpt");
    if (A->nnz > 0 && (!A->col || !A->val)) return fail(SELL_EINVAL, "sell_build: NULL col/val");
    if ((o->flags & SELL_BUILD_PERMUTE_COLS) && A->nrows != A->ncols)
        return fail(SELL_EINVAL, "sell_build: column permutation needs a square matrix");
    int64_t np = (A->nrows + o->C - 1) / o->C * (int64_t)o->C;
    if (np > 0x7FFFFFFFll) return fail(SELL_EINVAL, "sell_build: padded row count exceeds 2^31");
    return SELL_OK;
}

sell_status malformed(unsigned int err) {
    std::string m = "sell_build: malformed CRS:";
    if (err & kErrRpt0) m += " rpt[0] != 0;";
    if (err & kErrRptOrder) m += " rpt decreasing;";
    if (err & kErrRptEnd) m += " rpt[nrows] != nnz;";
    if (err & kErrRowLong) m += " row longer than 2^31-1;";
    if (err & kErrCol) m += " column index out of range;";
    return fail(SELL_EINVAL, m);
}

}  // namespace

sell_status build_format(const sell_csr *A, const sell_opts *o, cudaStream_t s, sell_matrix *h) {
    SELL_TRY(validate(A, o));
    const Allocator al = current_allocator();
    const int64_t N = A->nrows, nnz = A->nnz;
    const int C = o->C;
    const int64_t Nc = (N + C - 1) / C, Np = Nc * C;
    const size_t vin = A->val_type == SELL_F64 ? 8 : 4;

    // 1. the CRS arrays on the device
    DevBuf drpt, dcol, dval;
    const int64_t *rpt = A->rpt;
    const int32_t *col_in = A->col;
    const void *val_in = A->val;
    if (!A->on_device) {
        if (A->rpt[0] != 0 || A->rpt[N] != nnz)
            return fail(SELL_EINVAL, "sell_build: rpt[0] must be 0 and rpt[nrows] must be nnz");
        SELL_TRY(drpt.alloc(al, (N + 1) * sizeof(int64_t), s));
        SELL_CUDA_TRY(cudaMemcpyAsync(drpt.p, A->rpt, (N + 1) * sizeof(int64_t),
                                      cudaMemcpyHostToDevice, s));
        if (nnz > 0) {
            SELL_TRY(dcol.alloc(al, nnz * sizeof(int32_t), s));
            SELL_TRY(dval.alloc(al, nnz * vin, s));
            SELL_CUDA_TRY(cudaMemcpyAsync(dcol.p, A->col, nnz * sizeof(int32_t),
                                          cudaMemcpyHostToDevice, s));
            SELL_CUDA_TRY(cudaMemcpyAsync(dval.p, A->val, nnz * vin, cudaMemcpyHostToDevice, s));
        }
        rpt = drpt.as<int64_t>();
        col_in = dcol.as<int32_t>();
        val_in = dval.p;
    }

    // 2. row lengths + validation
    DevBuf rl, stats;
    SELL_TRY(stats.alloc(al, sizeof(BuildStats), s));
    SELL_CUDA_TRY(cudaMemsetAsync(stats.p, 0, sizeof(BuildStats), s));
    if (N > 0) {
        SELL_TRY(rl.alloc(al, N * sizeof(int32_t), s));
        k_rowlen<<<grid_for(N, 256, 152 * 4), 256, 0, s>>>(rpt, N, nnz, rl.as<int32_t>(), stats.as<BuildStats>());
        SELL_CUDA_TRY(cudaGetLastError());
    }
    BuildStats hs;
    SELL_CUDA_TRY(cudaMemcpyAsync(&hs, stats.p, sizeof(hs), cudaMemcpyDeviceToHost, s));
    SELL_CUDA_TRY(cudaStreamSynchronize(s));
    if (N == 0 && nnz != 0) hs.err |= kErrRptEnd;
    if (hs.err) return malformed(hs.err);

    // 3. sorting scope
    DevBuf perm;
    const bool sorted = o->sigma > 1 && N > 1;
    if (sorted) {
        SELL_TRY(perm.alloc(al, N * sizeof(int32_t), s));
        SELL_TRY(sort_windows(rl.as<int32_t>(), N, o->sigma, hs.max_rl, perm.as<int32_t>(), al, s));
    }

    // 4. chunk lengths (Eq. "max") and sorted row lengths
    DevBuf srl, cl, cs, inv, src;
    if (Np > 0) {
        SELL_TRY(srl.alloc(al, Np * sizeof(int32_t), s));
        SELL_TRY(cl.alloc(al, 2 * Nc * sizeof(int32_t), s));  // and the long rows per chunk
        SELL_TRY(src.alloc(al, Np * sizeof(int64_t), s));
        SELL_CUDA_TRY(cudaMemsetAsync(cl.p, 0, 2 * Nc * sizeof(int32_t), s));
    }
    const bool permute_cols = (o->flags & SELL_BUILD_PERMUTE_COLS) != 0;
    if (permute_cols && N > 0) SELL_TRY(inv.alloc(al, N * sizeof(int32_t), s));
    // (for the padded blocks of binary32 vectors, sell_internal.cuh)
    const int64_t near_step = C % 32 == 0 && nnz > 0 && o->store_type != SELL_F64 ? std::max<int64_t>(1, Np / 32 / kNearSlices) : 0;
    if (Np > 0) {
        int g = grid_for(Np, 256);
        k_chunk_len<<<g, 256, 0, s>>>(rl.as<int32_t>(), sorted ? perm.as<int32_t>() : nullptr, rpt, N, Np,
                                      C, srl.as<int32_t>(), src.as<int64_t>(), cl.as<int32_t>(), cl.as<int32_t>() + Nc,
                                      permute_cols ? inv.as<int32_t>() : nullptr, col_in, near_step,
                                      stats.as<BuildStats>());
        SELL_CUDA_TRY(cudaGetLastError());
    }
    // 5. chunk offsets, and the chunks that hold rows longer than kSeg.  The
    // scratch of sell_spmv_dot follows the offsets of a square matrix, ready
    // before the first product: allocated on first use, its clearing could be
    // recorded in a graph instead of done.
    const int64_t dot_words = N > 0 && N == A->ncols ? kDotRanges + 1 : 0;
    SELL_TRY(cs.alloc(al, (Nc + 1 + dot_words) * sizeof(int64_t), s));
    int64_t *dot_at = dot_words ? cs.as<int64_t>() + Nc + 1 : nullptr;
    DevBuf tile, lpos, ubase, wbase;
    ChunkSums total = {0, 0, 0, 0, 0};
    if (Nc > 0) {
        // tile sums, then the grand total; the block of tile t adds up the t
        // tile sums before it (at most 2048)
        const int64_t per = ((Nc + 2047) / 2048 + kScanThreads - 1) / kScanThreads * kScanThreads;
        const int64_t nt = (Nc + per - 1) / per;
        SELL_TRY(tile.alloc(al, (nt + 1) * sizeof(ChunkSums), s));
        SELL_TRY(lpos.alloc(al, Nc * sizeof(int64_t), s));
        SELL_TRY(ubase.alloc(al, Nc * sizeof(int64_t), s));
        SELL_TRY(wbase.alloc(al, Nc * sizeof(WorkBase), s));
        const int32_t *nlr = cl.as<int32_t>() + Nc;
        ChunkSums *tp = tile.as<ChunkSums>();
        k_chunk_reduce<<<(unsigned)nt, kScanThreads, 0, s>>>(cl.as<int32_t>(), nlr, Nc, per, C, tp);
        SELL_CUDA_TRY(cudaGetLastError());
        k_chunk_apply<<<(unsigned)nt, kScanThreads, 0, s>>>(cl.as<int32_t>(), nlr, Nc, per, C, tp, cs.as<int64_t>(),
                                                            lpos.as<int64_t>(), ubase.as<int64_t>(),
                                                            wbase.as<WorkBase>(), tp + nt,
                                                            dot_at ? dot_at + kDotRanges : nullptr);
        SELL_CUDA_TRY(cudaGetLastError());
        SELL_CUDA_TRY(cudaMemcpyAsync(&total, tp + nt, sizeof(total), cudaMemcpyDeviceToHost, s));
        SELL_CUDA_TRY(cudaStreamSynchronize(s));
    } else {
        SELL_CUDA_TRY(cudaMemsetAsync(cs.p, 0, sizeof(int64_t), s));
    }
    const int64_t stored = total.stored, nlong = total.nlong, nunits = total.nunits;
    DevBuf lchunk, lunit, cnt, cnt2, part, lrow, lmeta, lwork, lval, lcol;
    if (nlong > 0) {
        SELL_TRY(lchunk.alloc(al, nlong * sizeof(int32_t), s));
        SELL_TRY(lunit.alloc(al, nunits * sizeof(int2), s));
        SELL_TRY(lrow.alloc(al, (size_t)nlong * C * sizeof(int32_t), s));
        SELL_TRY(lmeta.alloc(al, (size_t)nlong * sizeof(LongMeta), s));
        if (total.nwork > 0) SELL_TRY(lwork.alloc(al, (size_t)total.nwork * sizeof(LongWork), s));
        if (total.npack > 0) {
            SELL_TRY(lval.alloc(al, (size_t)total.npack * kSeg * value_size(o->store_type), s));
            SELL_TRY(lcol.alloc(al, (size_t)total.npack * kSeg * sizeof(int32_t), s));
        }
        k_long_lists<<<(unsigned)((Nc + 7) / 8), 256, 0, s>>>(cl.as<int32_t>(), srl.as<int32_t>(),
                                                                  lpos.as<int64_t>(), ubase.as<int64_t>(),
                                                                  wbase.as<WorkBase>(), cs.as<int64_t>(), Nc, N, C,
                                                                  lchunk.as<int32_t>(), lunit.as<int2>(),
                                                                  lrow.as<int32_t>(), lmeta.as<LongMeta>(),
                                                                  lwork.as<LongWork>());
        SELL_CUDA_TRY(cudaGetLastError());
        SELL_TRY(cnt.alloc(al, nlong * C * sizeof(int32_t), s));
        SELL_CUDA_TRY(cudaMemsetAsync(cnt.p, 0, nlong * C * sizeof(int32_t), s));
        SELL_TRY(cnt2.alloc(al, (size_t)nunits * C * sizeof(int32_t), s));
        SELL_CUDA_TRY(cudaMemsetAsync(cnt2.p, 0, (size_t)nunits * C * sizeof(int32_t), s));
        SELL_TRY(part.alloc(al, (size_t)nunits * C * 8, s));
    }

    // 6. values and columns (the column range is checked on the way)
    DevBuf val, col, scol, sflag;
    bool pattern = false;
    const bool tiled = C % 32 == 0;
    const size_t vs = value_size(o->store_type);
    if (stored > 0) {
        SELL_TRY(val.alloc(al, stored * vs, s));
        SELL_TRY(col.alloc(al, stored * sizeof(int32_t), s));
        ScatterArgs a;
        a.src = src.as<int64_t>();
        a.col_in = col_in;
        a.val_in = val_in;
        a.inv = permute_cols ? inv.as<int32_t>() : nullptr;
        a.srl = srl.as<int32_t>();
        a.cl = cl.as<int32_t>();
        a.cs = cs.as<int64_t>();
        a.lchunk = lchunk.as<int32_t>();
        a.lunit = lunit.as<int2>();
        a.lrow = lrow.as<int32_t>();
        a.lwork = lwork.as<LongWork>();
        a.nunits = nunits;
        a.nlwork = total.nwork;
        a.lval = lval.p;
        a.lcol = lcol.as<int32_t>();
        a.N = N;
        a.Np = Np;
        a.ncols = A->ncols;
        a.C = C;
        a.val = val.p;
        a.col = col.as<int32_t>();
        a.scol = a.sflag = nullptr;
        if (tiled) {
            SELL_TRY(scol.alloc(al, (stored / 32 + 3 * (Np / 32) + 8) * sizeof(int32_t), s));
            SELL_TRY(sflag.alloc(al, Np / 32 * sizeof(int32_t), s));
            SELL_CUDA_TRY(cudaMemsetAsync(sflag.p, 1, Np / 32 * sizeof(int32_t), s));  // any non-zero word: a pattern
            a.scol = scol.as<int32_t>();
            a.sflag = sflag.as<int32_t>();
        }
        a.st = stats.as<BuildStats>();
        if (A->val_type == SELL_F64) SELL_TRY(launch_scatter<double>(a, o->store_type, s));
        else SELL_TRY(launch_scatter<float>(a, o->store_type, s));
        BuildStats end;
        SELL_CUDA_TRY(cudaMemcpyAsync(&end, a.st, sizeof(end), cudaMemcpyDeviceToHost, s));
        SELL_CUDA_TRY(cudaStreamSynchronize(s));
        if (end.err) return malformed(end.err);
        // The products take the offsets where they save column bytes: at least
        // half of the entries in slices with a pattern (a slice without one
        // reads its columns).
        unsigned long long nopat = 0;
        for (unsigned long long n : end.nopat) nopat += n;
        h->near = near_step > 0 && 2 * (int64_t)end.far * near_step <= Np / 32;
        h->local = tiled && nnz > 0 && 4 * ((unsigned long long)nnz - nopat) >= (unsigned long long)nnz;
        // The kernel loads offsets and prefetches values and columns in 16-byte units.
        pattern = tiled && 2 * nopat <= (unsigned long long)nnz &&
                  ((uintptr_t)val.p | (uintptr_t)col.p | (uintptr_t)scol.p) % 16 == 0;
    }
    if (!pattern) {
        scol.reset();
        sflag.reset();
    }
    SELL_CUDA_TRY(cudaStreamSynchronize(s));

    // 7. hand the arrays to the handle
    h->nrows = N;
    h->ncols = A->ncols;
    h->nnz = nnz;
    h->nchunks = Nc;
    h->stored = stored;
    h->sigma = o->sigma;
    h->max_rl = hs.max_rl;
    h->C = C;
    h->store_type = o->store_type;
    h->flags = o->flags;
    h->beta = stored > 0 ? (double)nnz / (double)stored : 1.0;
    if (N > 0 && nnz > 0) {
        double mean = (double)nnz / (double)N;
        double var = (double)hs.sumsq / (double)N - mean * mean;
        h->zeta = var > 0 ? std::sqrt(var) / mean : 0.0;
    } else {
        h->zeta = 0.0;
    }
    h->al = al;
    h->nlong = nlong;
    h->nunits = nunits;
    h->nlwork = total.nwork;
    h->part_k = nunits > 0 ? 1 : 0;
    h->device_bytes = val.bytes + col.bytes + cs.bytes + cl.bytes + srl.bytes + perm.bytes + lchunk.bytes +
                      lunit.bytes + cnt.bytes + cnt2.bytes + part.bytes + lrow.bytes + lmeta.bytes +
                      scol.bytes + sflag.bytes + lwork.bytes + lval.bytes + lcol.bytes;
    h->lwork = (LongWork *)lwork.release_ownership();
    h->lval = lval.release_ownership();
    h->lcol = (int32_t *)lcol.release_ownership();
    h->scol = (int32_t *)scol.release_ownership();
    h->sflag = (int32_t *)sflag.release_ownership();
    h->lchunk = (int32_t *)lchunk.release_ownership();
    h->lunit = (int2 *)lunit.release_ownership();
    h->lrow = (int32_t *)lrow.release_ownership();
    h->lmeta = (LongMeta *)lmeta.release_ownership();
    h->cnt = (int32_t *)cnt.release_ownership();
    h->cnt2 = (int32_t *)cnt2.release_ownership();
    h->part = part.release_ownership();
    h->val = val.release_ownership();
    h->col = (int32_t *)col.release_ownership();
    h->cs = (int64_t *)cs.release_ownership();
    h->dot_part = reinterpret_cast<double *>(dot_at);
    h->cl = (int32_t *)cl.release_ownership();
    h->srl = (int32_t *)srl.release_ownership();
    h->perm = (int32_t *)perm.release_ownership();
    return SELL_OK;
}

// The per-warp work split of the bulk-staged SpMV for nw warps (the per-chunk
// staged columns are computed on the first call).  Synchronises s.
sell_status bulk_plan(sell_matrix *h, int64_t nw, cudaStream_t s) {
    const int64_t Nc = h->nchunks;
    if (Nc >= INT32_MAX || nw >= (1 << 20)) return fail(SELL_EUNSUPPORTED, "bulk-staged SpMV: plan too large");
    const Allocator &al = h->al;
    if (!h->dstat) {
        void *p = al.get(sizeof(int32_t), s);
        if (!p) return fail(SELL_ENOMEM, "bulk plan allocation failed");
        h->dstat = static_cast<int32_t *>(p);
        SELL_CUDA_TRY(cudaMemsetAsync(h->dstat, 0, sizeof(int32_t), s));
    }
    DevBuf bss, bw;
    if (h->wsplit_n != nw && Nc > 0) {
        SELL_TRY(bw.alloc(al, Nc * sizeof(int32_t), s));
        if (!h->bsc) {
            void *p = al.get(Nc * sizeof(int32_t), s);
            if (!p) return fail(SELL_ENOMEM, "bulk plan allocation failed");
            h->bsc = static_cast<int32_t *>(p);
        }
        k_bulk_cols<<<grid_for(Nc * 32, 256, 152 * 16), 256, 0, s>>>(h->srl, h->nrows, Nc, h->C, h->bsc,
                                                                      bw.as<int32_t>());
        SELL_CUDA_TRY(cudaGetLastError());
    }
    if (h->wsplit_n != nw) {
        if (h->wsplit) {
            al.put(h->wsplit, s);
            h->wsplit = nullptr;
            h->wsplit_n = 0;
        }
        void *p = al.get((nw + 1) * sizeof(int32_t), s);
        if (!p) return fail(SELL_ENOMEM, "bulk plan allocation failed");
        h->wsplit = static_cast<int32_t *>(p);
        SELL_TRY(bss.alloc(al, (Nc + 1) * sizeof(int64_t), s));
        if (Nc > 0) {
            SELL_TRY(scan_exclusive<int32_t>(bw.as<int32_t>(), Nc, bss.as<int64_t>(), al, s));
        } else {
            SELL_CUDA_TRY(cudaMemsetAsync(bss.p, 0, sizeof(int64_t), s));
        }
        k_bulk_split<<<grid_for(nw + 1, 256), 256, 0, s>>>(bss.as<int64_t>(), Nc, nw, h->wsplit);
        SELL_CUDA_TRY(cudaGetLastError());
        h->wsplit_n = nw;
    }
    SELL_CUDA_TRY(cudaStreamSynchronize(s));
    return SELL_OK;
}

}  // namespace sell
