// sell_internal.cuh -- shared internals of the SELL-C-sigma CUDA library.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <mutex>
#include <string>
#include <vector>

#include "sell.h"
#include "sell_device.cuh"

namespace sell {

// ------------------------------------------------------------------ errors
void set_error(const std::string &msg);
sell_status fail(sell_status s, const std::string &msg);
sell_status cuda_fail(cudaError_t e, const char *what);

#define SELL_CUDA_TRY(expr)                                   \
    do {                                                      \
        cudaError_t _e = (expr);                              \
        if (_e != cudaSuccess) return ::sell::cuda_fail(_e, #expr); \
    } while (0)

#define SELL_TRY(expr)                         \
    do {                                       \
        sell_status _s = (expr);               \
        if (_s != SELL_OK) return _s;          \
    } while (0)

// --------------------------------------------------------------- allocator
struct Allocator {
    sell_alloc_fn alloc = nullptr;
    sell_free_fn release = nullptr;
    void *ctx = nullptr;
    void *get(size_t bytes, cudaStream_t s) const;
    void put(void *p, cudaStream_t s) const;
};
Allocator current_allocator();

// Device buffer released through the allocator it came from (RAII).
struct DevBuf {
    Allocator al;
    cudaStream_t stream = nullptr;
    void *p = nullptr;
    size_t bytes = 0;
    DevBuf() = default;
    DevBuf(const DevBuf &) = delete;
    DevBuf &operator=(const DevBuf &) = delete;
    ~DevBuf() { reset(); }
    sell_status alloc(const Allocator &a, size_t n, cudaStream_t s);
    void reset();
    void *release_ownership() { void *q = p; p = nullptr; bytes = 0; return q; }
    template <class T> T *as() const { return static_cast<T *>(p); }
};

inline size_t value_size(int t) { return t == SELL_F64 ? 8 : (t == SELL_F32 ? 4 : 2); }

// Accumulation of reduced-precision products: 0 binary32 chains, 1 Dot2 on
// every row, 2 Dot2 on rows longer than kSeg only.
inline int comp_mode(uint32_t flags) {
    if (flags & SELL_SPMV_COMPENSATED) return 1;
    return (flags & SELL_SPMV_COMPENSATED_LONG) ? 2 : 0;
}
constexpr uint32_t kCompFlags = SELL_SPMV_COMPENSATED | SELL_SPMV_COMPENSATED_LONG;
constexpr uint32_t kRhsFlags = SELL_SPMV_RHS_BLOCK4 | SELL_SPMV_RHS_BLOCK2 | SELL_SPMV_RHS_BLOCK1;

// The widest block of right-hand sides the flags allow (8 by default).
inline int max_rhs_block(uint32_t flags) {
    if (flags & SELL_SPMV_RHS_BLOCK1) return 1;
    if (flags & SELL_SPMV_RHS_BLOCK2) return 2;
    return (flags & SELL_SPMV_RHS_BLOCK4) ? 4 : 8;
}

// The next block of right-hand sides: the widest of 8, 4, 2, 1 that fits the
// remaining columns and the flags' limit.
inline int rhs_block(int rem, int maxw) {
    int kb = rem >= 8 ? 8 : rem >= 4 ? 4 : rem >= 2 ? 2 : 1;
    while (kb > maxw) kb >>= 1;
    return kb;
}

// Row pitches of X from here on (in elements) take 64-bit arithmetic: one
// column at a time, in kernels of their own (sell_rowdot.cuh, WidePitch).
constexpr int64_t kWidePitch = 1 << 28;

// Ranges of sell_spmv_dot (sell_dot.cu).
constexpr int kDotRanges = 1024;

// A block of 3 or of 5 to 7 right-hand sides of binary32 vectors (7 of
// binary64) runs as one of 4 or 8 on a copy of X with rows of that many
// values: one vector load per gathered row and one pass over the matrix, where
// the blocks 2 + 1 or 4 + 2 + 1 take a load per value and a pass each.  The
// kernels write the first `cols` columns, bits 4-7 of their vec argument (0:
// all).  Worth it where pad_pays says so.  Measured at k = 3 / 5 / 7, binary32: 1M lognormal rows 192 / 244 /
// 357 -> 105 / 129 / 139 us, 500,000 banded rows 50 / 80 / 116 -> 39 / 54 / 58
// us, 100^3 stencil 92 / 127 / 182 -> 64 / 81 / 85 us.  Binary64 pays for the
// columns that are not there with the FP64 pipe's time (100^3 stencil at k = 3
// 160 -> 213 us, at 5 273 -> 380 us) except at 7: lognormal 505 -> 352 us.
inline int pad_block(int rem, int maxw, bool f64) {
    if (rem == 3 && maxw >= 4 && !f64) return 4;
    return rem >= (f64 ? 7 : 5) && rem <= 7 && maxw >= 8 ? 8 : 0;
}

// How the kernels may load a row of X, or store a row of Y (base, row pitch
// ld elements of xs bytes): 2 with 32-byte vectors, 1 with 16-byte vectors,
// 0 value by value.  The kernels take X's in bits 0-1 and Y's in bits 2-3.
inline int x_vec(const void *X, int64_t ldx, size_t xs) {
    const uintptr_t a = (uintptr_t)X;
    const int64_t pitch = ldx * (int64_t)xs;
    if (a % 32 == 0 && pitch % 32 == 0) return 2;
    return (a % 16 == 0 && pitch % 16 == 0) ? 1 : 0;
}

}  // namespace sell

// ------------------------------------------------------------------ handle
struct sell_matrix {
    int64_t nrows = 0, ncols = 0, nnz = 0, nchunks = 0, stored = 0, sigma = 1, max_rl = 0;
    int32_t C = 32, store_type = SELL_F64;
    uint32_t flags = 0;
    double beta = 1.0, zeta = 0.0;
    int device = 0;
    int32_t block = 0, unroll = 0, pipeline = -1;  // 0, 0, -1: the library's choice (sell_spmv_impl.cuh)
    sell::Allocator al;
    // device arrays (owned)
    void *val = nullptr;       // stored elements of store_type
    int32_t *col = nullptr;    // stored
    int64_t *cs = nullptr;     // nchunks + 1
    int32_t *cl = nullptr;     // nchunks
    int32_t *srl = nullptr;    // nchunks * C, length of each sorted row
    int32_t *perm = nullptr;   // nrows, sorted -> original (null: identity)
    int32_t *lchunk = nullptr; // nlong chunks holding rows longer than kSeg
    // column offsets of slices with one column pattern (sell_build.cu
    // k_scatter_tiled): about stored / 32 offsets and one flag per 32 rows; null
    // unless most of the matrix lies in such slices
    int32_t *scol = nullptr, *sflag = nullptr;
    bool local = false;        // at least a quarter of the entries in such slices
    bool near = false;         // most slices' rows begin close together: X is read from cache (not binary64)
    int64_t nlong = 0;
    int2 *lunit = nullptr;     // nunits long-row work units {long chunk, segment}
    int32_t *lrow = nullptr;   // nlong * C lanes of each long chunk's long rows
    sell::LongMeta *lmeta = nullptr;  // nlong (sell_build.cu k_long_lists)
    int64_t nunits = 0;
    // long rows of single products (sell_long.cuh; null when C is no multiple of 32)
    sell::LongWork *lwork = nullptr;  // nlwork virtual warps
    int64_t nlwork = 0;
    void *lval = nullptr;      // entries of the virtual warps of chunks with few long rows,
    int32_t *lcol = nullptr;   //   kSeg of each per segment
    int32_t *cnt = nullptr;    // nlong * C per-row segment counters (zero at rest)
    int32_t *cnt2 = nullptr;   // nunits * C group counters of very long rows (zero at rest)
    void *part = nullptr;      // segment partials: nunits * C * part_k * 8 bytes
    int32_t part_k = 0;
    void *xpad = nullptr;      // padded copy of X (pad_block): ncols * 8 values, allocated on first use
    void *ppad = nullptr;      // segment partials of padded blocks: nunits * C * 8 * 8 bytes, allocated with xpad
    std::mutex pad_mu;         // held from the copy's launch to its product's, and for device_bytes
    // bulk-staged SpMV (launch mode 2), prepared by sell_set_launch
    int32_t *bsc = nullptr;    // nchunks staged columns per chunk
    int32_t *wsplit = nullptr; // wsplit_n + 1 per-warp chunk boundaries
    int64_t wsplit_n = 0;
    int32_t *dstat = nullptr;  // device status word: 1 after a bounded wait gave up
    int32_t bulk_grid = 0, bulk_warps = 0, bulk_ring = 0;
    mutable uint32_t expire_us = 0;  // one-shot test hook of sell_test_expire_wait (0: off),
                                     // consumed by the next bulk-staged launch
    double *dot_part = nullptr;  // range sums and block count of sell_spmv_dot, behind cs (square matrices)
    // host-io staging (lazily allocated): kIoSlots slots used in turn, so that
    // the copies of one call overlap the kernels of the previous ones when
    // calls alternate streams.  A slot is reused only after its result has
    // been copied out; with two slots that wait (the result copy of call i
    // before the input copy of call i + 2) bounds a call at half of the two
    // copies plus the kernel, with four the kernels set the pace.  done =
    // recorded after the slot's last device-to-host copy; kdone = recorded
    // after the latest host-io product's kernels.
    static constexpr int kIoSlots = 4;
    struct IoSlot {
        void *x = nullptr, *y = nullptr;
        size_t xb = 0, yb = 0;
        cudaEvent_t done = nullptr;
        bool used = false;
    } io[kIoSlots];
    int io_next = 0;
    cudaEvent_t kdone = nullptr;
    bool kdone_used = false;
    size_t device_bytes = 0;
};

struct sell_batch {
    struct Group {              // one launch: kernel variant, its products and units
        void *fn = nullptr;     // kernel entry
        void *params = nullptr; // host copy of the launch parameters (products and their unit ranges)
        bool lng = false;       // long rows (else short rows)
        int64_t nwork = 0;
        int32_t grid = 0;
    };
    int device = 0;
    sell::Allocator al;
    std::vector<void *> scratch;  // per-product segment scratch and counters
    std::vector<Group> groups;
    int64_t nwork = 0;
    int32_t nprod = 0;
    int32_t tile = 128;  // threads per block = rows (or segment threads) per work unit
    cudaStream_t last_stream = nullptr;  // stream of the latest sell_batch_run
    bool ran = false;
};

namespace sell {

// What a padded block costs is the copy of X, and what it saves are passes over
// the matrix and loads of X, which are cheap where neighbouring rows' columns lie
// close together (X lies in cache): there it takes 16 entries per column, 5 at
// seven vectors, elsewhere, and with long rows, which make every pass two
// launches, 3 (2).  Binary64 at seven pays the FP64 pipe for the
// eighth column, which patterns of more entries do not outweigh.  Measured in us, blocks /
// padded, 1M rows binary32 at three, five and seven vectors: patterns of 3
// entries 22 / 27, 23 / 37, 38 / 43; of 8 27 / 33, 31 / 43, 47 / 47; bands without a
// pattern of 5 28 / 37, 37 / 43, 54 / 46; 100^3 stencil
// 70 / 61, 93 / 76, 152 / 79; random columns, 2 per row 27 / 29, 37 / 39, 57 / 46;
// 3 per row 37 / 33, 47 / 43, 72 / 51.  Binary64 at seven: patterns of 5 entries
// 110 / 100, of 8 135 / 139, 100^3 stencil 360 / 386, but with long rows (dense
// 1000^2) 58 / 45.  Three columns trade one launch for another, which a small
// matrix of short rows is not worth (20^3 stencil 14.4 -> 16.2 us; 5000
// lognormal rows, with long ones, 41 -> 21 us).
inline bool pad_pays(const sell_matrix *h, int cols) {
    const bool f64 = h->store_type == SELL_F64;
    const int64_t least = h->near && !h->nunits && !f64 ? (cols == 7 ? 5 : 16) : (cols == 7 ? 2 : 3);
    if (h->ncols == 0 || h->nnz < least * h->ncols) return false;
    if (h->local && f64 && !h->nunits && h->nnz >= 8 * h->ncols) return false;
    return cols > 3 || h->nunits > 0 || h->nnz >= 500000;
}

// --------------------------------------------------------- launch entry points
// (defined in sell_spmv.cu / sell_build.cu / sell_batch.cu / sell_bench.cu)
sell_status launch_spmmv(sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy,
                         int32_t k, uint32_t flags, cudaStream_t s);
sell_status launch_block_with_scratch(const sell_matrix *h, const void *X, int64_t ldx, void *Y,
                                      int64_t ldy, int kb, uint32_t flags, void *part, int32_t *cnt,
                                      int32_t *cnt2, cudaStream_t s);
// dst (n x K, dense) = the first cols values of every row of X (n rows, ldx apart), zeros behind them.
cudaError_t launch_pad(const void *X, int64_t ldx, int64_t n, int cols, int K, size_t xs, void *dst, cudaStream_t s);
sell_status build_format(const sell_csr *A, const sell_opts *o, cudaStream_t s, sell_matrix *h);
sell_status bulk_plan(sell_matrix *h, int64_t nwarps, cudaStream_t s);
sell_status bulk_prepare(sell_matrix *h);
sell_status launch_dot(sell_matrix *h, const void *x, const void *y, double *out, cudaStream_t s);
// scratch: per item, batch_item_scratch() bytes of device memory (or NULL for
// items without long rows); NULL: the plan allocates its own.
sell_status batch_create(const sell_batch_item *items, int32_t n, cudaStream_t s, sell_batch *b,
                         void *const *scratch = nullptr);
size_t batch_item_scratch(const sell_matrix *h, int32_t k, uint32_t flags, size_t *counter_offset);
sell_status batch_run(sell_batch *b, int32_t grid, cudaStream_t s);
sell_status batch_set_tile(sell_batch *b, int32_t tile);
void batch_release(sell_batch *b, cudaStream_t s);
sell_status bench_read(const void *buf, size_t bytes, double *sink, int32_t grid, cudaStream_t s);
sell_status bench_fma64(double *sink, int32_t grid, int32_t iters, cudaStream_t s);
sell_status bench_gather(const void *x, int64_t n, double *sink, int32_t grid, int32_t iters, cudaStream_t s);
sell_status bench_gather4(const void *x, int64_t n, double *sink, int32_t grid, int32_t iters, cudaStream_t s);

}  // namespace sell
