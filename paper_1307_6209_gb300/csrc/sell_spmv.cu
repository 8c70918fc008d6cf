// sell_spmv.cu -- host side of the SELL-C-sigma SpMV / SpMMV: splits the
// right-hand sides into column blocks of 8/4/2/1, grows the long-row scratch
// and dispatches to the per-type kernels (sell_spmv_impl.cuh, instantiated in
// sell_spmv_f64.cu, sell_spmv_f32.cu, sell_spmv_bf16.cu).

#include <algorithm>
#include <mutex>

#include "sell_internal.cuh"

namespace sell {

// per-type entry points (sell_spmv_f64.cu / sell_spmv_f32.cu / sell_spmv_bf16.cu)
cudaError_t spmv_block_f64(const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int kb,
                           int acc, int vec, void *part, int32_t *cnt, int32_t *cnt2, cudaStream_t s);
cudaError_t spmv_block_f32(const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int kb,
                           int acc, int vec, int comp, void *part, int32_t *cnt, int32_t *cnt2, cudaStream_t s);
cudaError_t spmv_block_bf16(const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int kb,
                            int acc, int vec, int comp, void *part, int32_t *cnt, int32_t *cnt2, cudaStream_t s);

int bulk_blocks_per_sm_f64(const sell_matrix *h, int W, int R);
int bulk_blocks_per_sm_f32(const sell_matrix *h, int W, int R);
int bulk_blocks_per_sm_bf16(const sell_matrix *h, int W, int R);

namespace {

cudaError_t dispatch(const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int kb, int acc,
                     int vec, int comp, void *part, int32_t *cnt, int32_t *cnt2, cudaStream_t s) {
    switch (h->store_type) {
        case SELL_F64: return spmv_block_f64(h, X, ldx, Y, ldy, kb, acc, vec, part, cnt, cnt2, s);
        case SELL_F32: return spmv_block_f32(h, X, ldx, Y, ldy, kb, acc, vec, comp, part, cnt, cnt2, s);
        default: return spmv_block_bf16(h, X, ldx, Y, ldy, kb, acc, vec, comp, part, cnt, cnt2, s);
    }
}

// One thread per value of the padded rows: reads and writes run along the rows.
template <class T>
__global__ void __launch_bounds__(256) k_pad(const T *__restrict__ X, int64_t ldx, int64_t n, int cols, int K,
                                             T *__restrict__ dst) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n * K; i += stride) {
        const int64_t row = K == 4 ? i >> 2 : i >> 3;
        const int q = (int)(i & (K - 1));
        dst[i] = q < cols ? X[row * ldx + q] : T(0);
    }
}

bool grow_part(sell_matrix *h, int need, cudaStream_t s) {
    void *p = h->al.get((size_t)h->nunits * h->C * need * 8, s);
    if (!p) return false;
    h->al.put(h->part, s);
    h->part = p;
    h->part_k = need;
    return true;
}

// Memory for padded blocks: the copy of X and a long-row scratch of their own,
// once per handle and for the widest block.  Neither ever moves, and h->part
// does not grow for a padded block, so the pointers in a captured graph stay
// good whatever widths run after it.  Allocates nothing while the stream is
// captured (the blocks 4, 2, 1 need neither).
bool make_pad(sell_matrix *h, cudaStream_t s) {
    const bool part = h->nunits > 0 && !h->ppad;
    if (h->xpad && !part) return true;
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    if (st != cudaStreamCaptureStatusNone) return false;
    auto take = [&](void *&p, size_t bytes) {
        if (!p && (p = h->al.get(bytes, s))) h->device_bytes += bytes;
        return p != nullptr;
    };
    if (part && !take(h->ppad, (size_t)h->nunits * h->C * 8 * 8)) return false;
    return take(h->xpad, (size_t)h->ncols * 8 * (h->store_type == SELL_F64 ? 8 : 4));
}

}  // namespace

cudaError_t launch_pad(const void *X, int64_t ldx, int64_t n, int cols, int K, size_t xs, void *dst, cudaStream_t s) {
    const unsigned grid = (unsigned)std::min<int64_t>((n * K + 255) / 256, 152 * 64);
    if (xs == 8)
        k_pad<double><<<grid, 256, 0, s>>>(static_cast<const double *>(X), ldx, n, cols, K, static_cast<double *>(dst));
    else
        k_pad<float><<<grid, 256, 0, s>>>(static_cast<const float *>(X), ldx, n, cols, K, static_cast<float *>(dst));
    return cudaGetLastError();
}

// Splits k into kernel blocks of 8, 4, 2, 1 columns, at most the flags' block
// width, and odd numbers of last columns into one padded block (every column
// keeps the same per-row operation order, so the split does not change any
// result).  The segment scratch grows on the first
// product with a wider block.
sell_status launch_spmmv(sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy,
                         int32_t k, uint32_t flags, cudaStream_t s) {
    if (h->nrows == 0) return SELL_OK;
    const int maxw = ldx < kWidePitch ? max_rhs_block(flags) : 1;
    const size_t xs = h->store_type == SELL_F64 ? 8 : 4;
    const int last = k % 8, odd = pad_block(last, maxw, h->store_type == SELL_F64), plain = rhs_block(k, maxw);
    // Host threads may issue products of one handle on one stream: another
    // thread's copy must not come between this one's copy and its product.
    std::unique_lock<std::mutex> lock(h->pad_mu, std::defer_lock);
    if (odd && pad_pays(h, last)) lock.lock();
    const bool pad = lock.owns_lock() && make_pad(h, s);
    const int need = pad && k < 8 ? 0 : plain;
    if (h->nunits > 0 && need > h->part_k && !grow_part(h, need, s))
        return fail(SELL_ENOMEM, "segment scratch allocation failed");
    const int acc = (flags & SELL_SPMV_ACCUMULATE) ? 1 : 0;
    const int comp = comp_mode(flags);
    int32_t done = 0;
    while (done < k) {
        const int rem = k - done;
        const char *Xb = static_cast<const char *>(X) + (size_t)done * xs;
        char *Yb = static_cast<char *>(Y) + (size_t)done * xs;
        cudaError_t e;
        if (pad && rem == last) {
            e = launch_pad(Xb, ldx, h->ncols, rem, odd, xs, h->xpad, s);
            if (e == cudaSuccess)
                e = dispatch(h, h->xpad, odd, Yb, ldy, odd, acc, x_vec(h->xpad, odd, xs) | (rem << 4), comp, h->ppad,
                             h->cnt, h->cnt2, s);
            if (e != cudaSuccess) return cuda_fail(e, "SpMV kernel launch");
            break;
        }
        const int kb = rhs_block(rem, maxw);
        int vec = x_vec(Xb, ldx, xs) | (x_vec(Yb, ldy, xs) << 2);
        e = dispatch(h, Xb, ldx, Yb, ldy, kb, acc, vec, comp, nullptr, nullptr, nullptr, s);
        if (e != cudaSuccess) return cuda_fail(e, "SpMV kernel launch");
        done += kb;
    }
    return SELL_OK;
}

// One column block of up to 8 right-hand sides with the given segment scratch
// `part` (nunits * C * kb * 8 bytes) and zeroed counters `cnt` (nlong * C) and
// `cnt2` (nunits * C).
sell_status launch_block_with_scratch(const sell_matrix *h, const void *X, int64_t ldx, void *Y,
                                      int64_t ldy, int kb, uint32_t flags, void *part, int32_t *cnt,
                                      int32_t *cnt2, cudaStream_t s) {
    const int acc = (flags & SELL_SPMV_ACCUMULATE) ? 1 : 0;
    const int comp = comp_mode(flags);
    const size_t xs = h->store_type == SELL_F64 ? 8 : 4;
    const int vec = x_vec(X, ldx, xs) | (x_vec(Y, ldy, xs) << 2);
    cudaError_t e = dispatch(h, X, ldx, Y, ldy, kb, acc, vec, comp, part, cnt, cnt2, s);
    if (e != cudaSuccess) return cuda_fail(e, "SpMV kernel launch");
    return SELL_OK;
}

// Launch shape and work split of the bulk-staged SpMV for the handle's
// block (warps per block) and unroll (slots per warp: 1, 2, 3, 4 for unroll
// 1, 2, 4, 8; fewer if shared memory does not hold them): one persistent
// wave, every SM filled with as many blocks as fit.
sell_status bulk_prepare(sell_matrix *h) {
    h->bulk_grid = 0;  // the bulk kernel stays off until the plan below exists
    if (h->C != 32 && h->C != 64 && h->C != 128)
        return fail(SELL_EUNSUPPORTED, "bulk-staged SpMV needs C = 32, 64 or 128");
    // bulk copies need 16-byte aligned sources (chunk offsets are multiples of C)
    if (((uintptr_t)h->val | (uintptr_t)h->col | (uintptr_t)h->srl) % 16 != 0)
        return fail(SELL_EUNSUPPORTED, "bulk-staged SpMV needs 16-byte aligned format arrays");
    const int W = (h->block ? h->block : 256) / 32;
    const int u = h->unroll ? h->unroll : 4;
    int R = u >= 8 ? 4 : (u >= 4 ? 3 : (u >= 2 ? 2 : 1));
    int bps = 0;
    for (; R >= 1; --R) {
        switch (h->store_type) {
            case SELL_F64: bps = bulk_blocks_per_sm_f64(h, W, R); break;
            case SELL_F32: bps = bulk_blocks_per_sm_f32(h, W, R); break;
            default: bps = bulk_blocks_per_sm_bf16(h, W, R); break;
        }
        if (bps > 0) break;
    }
    if (bps <= 0) return fail(SELL_EUNSUPPORTED, "bulk-staged SpMV: the block does not fit on an SM");
    int nsm = 0;
    SELL_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, h->device));
    const int grid = nsm * bps;
    SELL_TRY(bulk_plan(h, (int64_t)grid * W, nullptr));
    h->bulk_grid = grid;
    h->bulk_warps = W;
    h->bulk_ring = R;
    return SELL_OK;
}

}  // namespace sell
