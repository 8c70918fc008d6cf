// sell_device.cuh -- the constants and device helpers that the SpMV kernels'
// arithmetic and memory behaviour depend on (kept apart from the host-side
// internals so that a change here is a change of the kernels).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace sell {
// Entries per segment of a long row.  Part of the numerics: a row longer than
// kSeg is summed segment by segment (sell_rowdot.cuh), so changing it changes
// the rounding of long rows.
constexpr int kSeg = 64;
// Segments per group of the two-level fold of very long rows (more than
// kSeg * kSuper = 16384 entries); also part of the numerics.
constexpr int kSuper = 256;

// Where the column offsets of a slice (32 rows) begin in scol: every slice
// takes its chunk's width, and starts at a multiple of four values so that
// four offsets are one 16-byte load.  The three values of slack per slice
// make room for the rounding: (a + 3g + 3) & ~3 grows by at least the width
// from one slice to the next.
__host__ __device__ __forceinline__ int64_t offset_start(int64_t cs0, int32_t width, int s, int64_t slice) {
    return ((cs0 >> 5) + (int64_t)s * width + 3 * slice + 3) & ~(int64_t)3;
}

// A virtual warp of the long rows (sell_long.cuh): long chunk lc = chunk c,
// whose first partial slot is u0 and which has nseg segments per row.
// m < 0: segment i / (C / 32) of 32 neighbouring rows; else the 32 segments
// from number 32 i of the chunk's m long rows, one row after another (fewer in
// the last).  base: where lane 0's first entry is.  (8-byte aligned at most, here and below: an
// allocator's memory need not be aligned for more.)
struct LongWork {
    int32_t lc, c, nseg, m;
    int64_t base;
    int32_t i, u0;
};

// A long chunk's long rows, how its units take them (0: a unit thread per lane, 1: its
// rows' segments one after another), and its segments per row.
struct LongMeta {
    int32_t m, mode, nseg;
};
static_assert(alignof(LongWork) <= 8 && alignof(LongMeta) <= 8, "an allocator's memory is 8-byte aligned");

// --------------------------------------------------------- device helpers
// Streaming loads for data touched once per product (val/col): do not allocate
// in L1 and mark the L2 lines evict-first, so that the gathered vector x keeps
// its place in L2.
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// Where `ask` holds, ask L2 for `bytes` (a multiple of 16) at p (16-byte
// aligned), one request.  A predicated instruction and not a branch: behind a
// branch that one lane takes, the warp can stay split, and what follows is
// issued twice (the column-pattern kernels, which ask with one lane: with the
// slice's flag loaded ahead of the branch 271 us on the 150^3 stencil binary32
// at eight vectors, behind it 183, predicated 166; 187^3 bfloat16 181, 153, 145).
__device__ __forceinline__ void prefetch_l2(bool ask, const void *p, uint32_t bytes, uint64_t pol) {
    asm volatile(
        "{\n"
        ".reg .pred ask;\n"
        "setp.ne.s32 ask, %3, 0;\n"
        "@ask cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;\n"
        "}" ::"l"(p), "r"(bytes), "l"(pol), "r"((int)ask));
}

__device__ __forceinline__ double ld_stream(const double *ptr, uint64_t pol) {
    double v;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.f64 %0, [%1], %2;"
                 : "=d"(v) : "l"(ptr), "l"(pol));
    return v;
}
__device__ __forceinline__ float ld_stream(const float *ptr, uint64_t pol) {
    float v;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.f32 %0, [%1], %2;"
                 : "=f"(v) : "l"(ptr), "l"(pol));
    return v;
}
__device__ __forceinline__ int32_t ld_stream(const int32_t *ptr, uint64_t pol) {
    int32_t v;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.s32 %0, [%1], %2;"
                 : "=r"(v) : "l"(ptr), "l"(pol));
    return v;
}
__device__ __forceinline__ __nv_bfloat16 ld_stream(const __nv_bfloat16 *ptr, uint64_t pol) {
    unsigned short v;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.b16 %0, [%1], %2;"
                 : "=h"(v) : "l"(ptr), "l"(pol));
    return __ushort_as_bfloat16(v);
}

}  // namespace sell
