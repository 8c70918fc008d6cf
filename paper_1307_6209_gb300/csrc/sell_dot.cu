// sell_dot.cu -- the dot product x . y that follows an SpMV in a Krylov step
// (the p . Ap of conjugate gradients), in binary64 and in a fixed order.
//
// The sum does not depend on the format, the launch or the run: element i of
// the n-vector belongs to range b = i / ceil(n / kDotBlocks) of kDotBlocks
// contiguous ranges; inside a range, slot t of kDotThreads adds elements
// t, t + kDotThreads, ... in that order (fma of the binary64 products), the
// slots are then added in a fixed tree, and the kDotBlocks range sums in a
// fixed tree too.  y is read right after the SpMV wrote it, mostly from L2.
//
// One launch, of two forms by the length of a range: a warp per range (up to
// kDotThreads elements, one per slot) or a block per range.  The block that
// finishes last adds the range sums.  The launch is a programmatic dependent
// of the product's: it is brought up and loads x while that runs, and waits
// for its end.  Before, the ranges and the final sum were two launches, with
// a block of 256 threads for every range: 12 us from the product's end to the
// dot on the 64 x 64 Laplacian, now 5.  A warp's binary64 instruction takes 64
// cycles of its scheduler's FP64 pipe whatever the lanes do, so slots that a
// range does not reach are left out of the additions, and one block for all
// ranges of a short vector would be slower (7 us).
#include "sell_internal.cuh"

namespace sell {
namespace {

constexpr int kDotBlocks = kDotRanges;
constexpr int kDotThreads = 256;

__device__ __forceinline__ double as_f64(double v) { return v; }
__device__ __forceinline__ double as_f64(float v) { return (double)v; }
__device__ __forceinline__ void wait_for_product() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Slot a of a range of len elements and its partner `other` = slot at: a
// partner beyond the range is +0, whose addition only turns -0 into +0.
__device__ __forceinline__ void add_slot(double &a, double other, int at, int len) {
    if (at < len) a += other;
    else if (__double_as_longlong(a) == (long long)0x8000000000000000ull) a = 0.0;
}

// The sum of red[0 .. n) (n a power of two, at least 64): pairs n / 2 apart,
// then n / 4, ...  All threads of the block call; thread 0 has the result.
__device__ __forceinline__ double tree(double *red, int n) {
    for (int w = n / 2; w >= 32; w >>= 1) {
        __syncthreads();
        for (int i = threadIdx.x; i < w; i += blockDim.x) red[i] += red[i + w];
    }
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < 32) {
        s = red[threadIdx.x];
        for (int w = 16; w > 0; w >>= 1) s += __shfl_down_sync(0xffffffffu, s, w);
    }
    return s;
}

// The block that completes the range sums adds them (count: blocks done, zero
// between products).
__device__ __forceinline__ void finish(const double *part, int *count, double *red, double *out) {
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(count, 1) == (int)gridDim.x - 1;
        if (last) __threadfence();
    }
    __syncthreads();
    if (!last) return;
    for (int i = threadIdx.x; i < kDotBlocks; i += blockDim.x) red[i] = __ldcg(part + i);
    const double v = tree(red, kDotBlocks);
    if (threadIdx.x == 0) {
        *out = v;
        *count = 0;
    }
}

// Q: slots per lane that a range of len elements can reach (32 Q >= len).
template <class T, int Q>
__global__ void __launch_bounds__(kDotThreads) k_dot_warps(const T *__restrict__ x, const T *y, int n, double *part,
                                                           int *count, double *__restrict__ out) {
    __shared__ double red[kDotBlocks];
    constexpr int S = kDotThreads / 32;  // slots per lane: lane, lane + 32, ...
    const int len = (n + kDotBlocks - 1) / kDotBlocks, lane = threadIdx.x & 31;
    const int b = blockIdx.x * S + (threadIdx.x >> 5);  // the block's warps take S ranges
    const int b0 = b * len, m = min(len, n - b0);
    T xv[Q], yv[Q];
    double s[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) xv[q] = x[lane + 32 * q < m ? b0 + lane + 32 * q : 0];
    wait_for_product();
#pragma unroll
    for (int q = 0; q < Q; ++q) yv[q] = y[lane + 32 * q < m ? b0 + lane + 32 * q : 0];
#pragma unroll
    for (int q = 0; q < Q; ++q) s[q] = lane + 32 * q < m ? fma(as_f64(xv[q]), as_f64(yv[q]), 0.0) : 0.0;
#pragma unroll
    for (int w = S / 2; w > 0; w >>= 1)
#pragma unroll
        for (int q = 0; q < w && q < Q; ++q) add_slot(s[q], q + w < Q ? s[q + w < Q ? q + w : 0] : 0.0, lane + 32 * (q + w), q + w < Q ? len : 0);
    double v = s[0];
    for (int w = 16; w > 0; w >>= 1) v += __shfl_down_sync(0xffffffffu, v, w);
    if (lane == 0) part[b] = v;
    finish(part, count, red, out);
}

template <class T>
__global__ void __launch_bounds__(kDotThreads) k_dot_blocks(const T *__restrict__ x, const T *y, int64_t n,
                                                            double *part, int *count, double *__restrict__ out) {
    __shared__ double red[kDotBlocks];
    const int64_t len = (n + kDotBlocks - 1) / kDotBlocks;
    const int64_t b0 = blockIdx.x * len, b1 = min(n, b0 + len);
    wait_for_product();
    double s = 0.0;
    for (int64_t i = b0 + threadIdx.x; i < b1; i += 4 * kDotThreads) {  // four loads in flight
        double a[4], c[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool in = i + q * kDotThreads < b1;
            a[q] = in ? as_f64(x[i + q * kDotThreads]) : 0.0;
            c[q] = in ? as_f64(y[i + q * kDotThreads]) : 0.0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i + q * kDotThreads < b1) s = fma(a[q], c[q], s);
    }
    red[threadIdx.x] = s;
    const double v = tree(red, kDotThreads);
    if (threadIdx.x == 0) part[blockIdx.x] = v;
    finish(part, count, red, out);
}

template <class T>
cudaError_t run_dot(sell_matrix *h, const T *x, const T *y, double *out, cudaStream_t s) {
    const int64_t n = h->nrows;
    int *count = reinterpret_cast<int *>(h->dot_part + kDotBlocks);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cfg.blockDim = dim3(kDotThreads);
    if (n <= kDotBlocks * kDotThreads) {
        const int64_t len = (n + kDotBlocks - 1) / kDotBlocks;
        auto kern = len <= 32 ? k_dot_warps<T, 1> : len <= 64 ? k_dot_warps<T, 2> : len <= 128 ? k_dot_warps<T, 4>
                                                                                            : k_dot_warps<T, 8>;
        cfg.gridDim = dim3(kDotBlocks / (kDotThreads / 32));
        return cudaLaunchKernelEx(&cfg, kern, x, y, (int)n, h->dot_part, count, out);
    }
    cfg.gridDim = dim3(kDotBlocks);
    return cudaLaunchKernelEx(&cfg, k_dot_blocks<T>, x, y, n, h->dot_part, count, out);
}

}  // namespace

sell_status launch_dot(sell_matrix *h, const void *x, const void *y, double *out, cudaStream_t s) {
    const cudaError_t e = h->store_type == SELL_F64
                              ? run_dot(h, static_cast<const double *>(x), static_cast<const double *>(y), out, s)
                              : run_dot(h, static_cast<const float *>(x), static_cast<const float *>(y), out, s);
    if (e != cudaSuccess) return cuda_fail(e, "dot kernel launch");
    return SELL_OK;
}

}  // namespace sell
