// sell_spmv_impl.cuh -- the SpMV / SpMMV kernel template and its launch
// helpers, included by one translation unit per value type
// (sell_spmv_f64.cu, sell_spmv_f32.cu, sell_spmv_bf16.cu).
//
// Mapping (Sec. 3.4, "Sliced ELLR-T"; Sec. 5: one thread per row): thread r
// handles sorted row r = c*C + l and walks its own row length over
// val[cs[c] + j*C + l] -- for a fixed j the C threads of a chunk read C
// consecutive elements, so the loads of val/col are coalesced when C is a
// multiple of 32, and no thread loads padding.  Rows longer than kSeg are
// cut into kSeg-entry segments, which a kernel of their own multiplies ahead
// of the short rows (sell_long.cuh).
// The result goes to y[perm[r]] (original order) or y[r] (permuted space).
//
// Memory behaviour: val/col are read once per product (L1 no-allocate, L2
// evict-first); x is gathered through the read-only path and stays
// L2-resident; U entries of a row are loaded per step (the last, partial
// group predicated), so each thread keeps up to 2U streaming loads and U
// gathers in flight.
#pragma once

#include <type_traits>

#include "sell_long.cuh"
#include "sell_rowdot.cuh"
#include "sell_spmv_bulk.cuh"

namespace sell {
namespace spmv_impl {


#define SELL_SPMMV_PARAMS                                                                              \
    const VT *__restrict__ val, const int32_t *__restrict__ col, const int64_t *__restrict__ cs,      \
        const int32_t *__restrict__ srl, const int32_t *__restrict__ perm, const Pattern pt,          \
        const typename XType<VT>::T *__restrict__ X, LD ldx, typename XType<VT>::T *Y, int64_t ldy,    \
        int64_t N, int C, int accumulate, int vec, int after_long
#define SELL_SPMMV_ARGS val, col, cs, srl, perm, pt, X, ldx, Y, ldy, N, C, accumulate, vec, after_long

// The rows of at most kSeg entries, one thread per row.  after_long: the long
// rows' kernel (sell_long.cuh) runs ahead of this one, which ends only once
// that has ended: the warps past the last row wait for it (launch_short adds a
// block of them, so that there are some).  A warp with rows of its own does
// not: they would be multiplied after the wait (unsorted lognormal rows
// binary64 at one / eight vectors, 2000 rows 20.5 / 53 us then, 14.4 / 35 us
// so; 50,000 rows 38 / 120 and 27 / 100 us).
template <class VT, int K, int U, bool PIPE, class Acc, bool PAT, int CT, class LD>
__device__ __forceinline__ void spmmv_body(SELL_SPMMV_PARAMS) {
    using XT = typename XType<VT>::T;
    dependents_may_start();  // a dot product's launch (sell_dot.cu)
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= N) {
        if (after_long && r - (threadIdx.x & 31) >= N) wait_for_predecessor();
        return;
    }
    short_row<VT, XT, K, U, PIPE, Acc, PAT, CT>(val, col, cs, srl, perm, pt, X, ldx, Y, ldy, C, (uint32_t)r, accumulate,
                                            vec, l2_evict_first_policy());
}

template <class VT, int K, int U, bool PIPE, class Acc, class LD = Pitch>
__global__ void __launch_bounds__(512) k_spmmv(SELL_SPMMV_PARAMS) {
    spmmv_body<VT, K, U, PIPE, Acc, false, 0, LD>(SELL_SPMMV_ARGS);
}

// Occupancy: the one-vector kernel asks for 4 resident blocks of 512 threads,
// i.e. 32 registers -- every warp slot of the SM at any block size.  Its
// pipelined forms would otherwise take 39-40
// registers (48 of 64 warps); capped they spill 12-28 bytes and still run
// faster, measured on the 200^3 stencil: binary64 (unroll 2, pipelined)
// 467 -> 420 us, the best launch overall (425.5 us before); binary32
// (unroll 4, pipelined) 319 -> 295 us; bfloat16 unchanged.  The other
// kernels keep the allocation ptxas picks (capping the wider ones spills
// hundreds of bytes).
template <class VT, int U, bool PIPE, class Acc, int CT = 0, class LD = Pitch>
__global__ void __launch_bounds__(512, 4) k_spmv_short(SELL_SPMMV_PARAMS) {
    spmmv_body<VT, 1, U, PIPE, Acc, false, CT, LD>(SELL_SPMMV_ARGS);
}

template <class VT, int K, int U, bool PIPE, int MINB, class Acc, class LD = Pitch>
__global__ void __launch_bounds__(512, MINB) k_spmmv_pattern(SELL_SPMMV_PARAMS) {
    spmmv_body<VT, K, U, PIPE, Acc, true, 0, LD>(SELL_SPMMV_ARGS);
}

#undef SELL_SPMMV_PARAMS
#undef SELL_SPMMV_ARGS

// Where the column patterns are used: several binary64 vectors at once wait
// for the FP64 pipe, and the pattern kernels' registers cost more than the
// columns do (100^3 stencil at two vectors 101 us, 94 us without).
template <class VT, int K>
constexpr bool pattern_width() {
    return K == 1 || sizeof(VT) < 8;
}

template <class VT, int K, class AccL>
cudaError_t run_long(const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int acc, int vec,
                     void *part, int32_t *cnt, int32_t *cnt2, cudaStream_t s) {
    using XT = typename XType<VT>::T;
    const bool wide = ldx >= kWidePitch, pat = pattern_width<VT, K>() && h->scol != nullptr && !wide;
    const LongArgs a = long_args(h, pat);
    const VT *val = static_cast<const VT *>(h->val);
    const VT *lval = static_cast<const VT *>(h->lval);
    const XT *x = static_cast<const XT *>(X);
    XT *y = static_cast<XT *>(Y);
    constexpr int U = long_shape<VT, K>().unroll;
    constexpr bool P = long_shape<VT, K>().pipe;
    const unsigned blocks = (unsigned)((long_threads(h) + kLongThreads - 1) / kLongThreads);
    if constexpr (K == 1) {
        if (wide) {
            k_long<VT, 1, 1, false, AccL, false, WidePitch><<<blocks, kLongThreads, 0, s>>>(
                val, lval, a, part, cnt, cnt2, x, ldx, y, ldy, acc, vec);
            return cudaGetLastError();
        }
    }
    auto kern = k_long<VT, K, U, P, AccL, false, Pitch>;
    if constexpr (pattern_width<VT, K>()) {
        if (pat) kern = k_long<VT, K, U, P, AccL, true, Pitch>;
    }
    if constexpr (K == 4 && sizeof(VT) == 8) {
        // with most of the entries, in full segments, the kernel has the chip
        // to itself, and the loads in flight are worth the registers: dense
        // 3000^2 94 us with unroll 2, 86 us so.  1M sorted lognormal rows, a
        // third of the entries here, 113 and 115 us; 60,000 in windows of 256,
        // most lanes of whose virtual warps are idle, 39 and 46 us
        const int64_t held = long_threads(h) * kSeg;  // entries of so many full segments
        if (2 * held > h->nnz && 4 * held <= 5 * h->nnz) kern = k_long<VT, K, 4, true, AccL, false, Pitch>;
    }
    kern<<<blocks, kLongThreads, 0, s>>>(val, lval, a, part, cnt, cnt2, x, Pitch{(int32_t)(ldx * sizeof(XT))}, y, ldy,
                                         acc, vec);
    return cudaGetLastError();
}

// Threads per block unless sell_set_launch says otherwise: a block's warps
// leave the SM together, so the small ones lose less to rows of different
// lengths (2M sorted lognormal rows binary64, unroll 4: block 128 132.7 us,
// 256 137.4 us, 512 141.7 us; 64 gains nothing more).
constexpr int kBlock = 128;
constexpr int64_t kFewRows = 152 * 2048;  // the chip's threads

// One launch of a short-row kernel, behind the long rows' where there are any.
template <class VT, class LD, class Kernel>
cudaError_t launch_short_with(Kernel kern, const sell_matrix *h, const void *X, LD ldx, void *Y, int64_t ldy, int acc,
                              int vec, cudaStream_t s) {
    using XT = typename XType<VT>::T;
    const VT *val = static_cast<const VT *>(h->val);
    const int32_t *perm = (h->flags & SELL_BUILD_PERMUTE_COLS) ? nullptr : h->perm;
    const XT *x = static_cast<const XT *>(X);
    XT *y = static_cast<XT *>(Y);
    const Pattern pt{h->scol, h->sflag, h->cl};
    const int block = h->block ? h->block : kBlock;
    const unsigned blocks = (unsigned)((h->nrows + block - 1) / block);
    if (!h->nunits) {
        kern<<<blocks, block, 0, s>>>(val, h->col, h->cs, h->srl, perm, pt, x, ldx, y, ldy, h->nrows, h->C, acc, vec,
                                         0);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks + 1);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, val, static_cast<const int32_t *>(h->col),
                              static_cast<const int64_t *>(h->cs), static_cast<const int32_t *>(h->srl), perm, pt, x,
                              ldx, y, ldy, h->nrows, (int)h->C, acc, vec, 1);
}
template <class VT, class Kernel>
cudaError_t launch_short(Kernel kern, const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int acc,
                         int vec, cudaStream_t s) {
    const Pitch p{(int32_t)(ldx * (int64_t)sizeof(typename XType<VT>::T))};
    return launch_short_with<VT, Pitch>(kern, h, X, p, Y, ldy, acc, vec, s);
}

template <class VT, int K, int U, bool PIPE, class Acc>
cudaError_t run(const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int acc, int vec,
                cudaStream_t s) {
    if constexpr (K == 1) return launch_short<VT>(k_spmv_short<VT, U, PIPE, Acc>, h, X, ldx, Y, ldy, acc, vec, s);
    else return launch_short<VT>(k_spmmv<VT, K, U, PIPE, Acc>, h, X, ldx, Y, ldy, acc, vec, s);
}

// Matrices whose slices have column patterns: the product reads the values
// and one offset per 32 entries instead of 32 columns, and the gathers no
// longer wait for streamed columns.  Bound: HBM for the values (binary64 at
// one vector: the FP64 pipe, 348 us on the 200^3 stencil).  Measured, block
// 128, before -> after: 200^3 stencil binary64 423 -> 374 us; 187^3 binary32
// 219 -> 167 us and bfloat16 212 -> 145 us (best launch before); 150^3
// binary32 at k = 4 / 8 206 (k = 8) -> 137 / 166 us; dense 3000^2 binary32
// 18.8 -> 16.6 us.  Unroll, pipelining and resident blocks per width were
// swept on these; more loads in flight per thread cost registers, and the
// kernel loses more warps than it gains loads (binary64 with unroll 8:
// 437 us; k = 8 with 3 blocks: 438 us, spills; k = 8 with unroll 2 168 us, not
// pipelined 191 us; one binary32 vector with unroll 8 168 us, bfloat16 148 us).
template <class VT, int K, class Acc>
cudaError_t run_pattern(const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int acc, int vec,
                        cudaStream_t s) {
    constexpr bool F64 = sizeof(VT) == 8;
    auto pick = [&]() {
        if constexpr (K == 1) return k_spmmv_pattern<VT, K, F64 ? 2 : 4, F64, 4, Acc>;
        else if constexpr (K == 2) return k_spmmv_pattern<VT, K, 4, true, 3, Acc>;
        else if constexpr (K == 4) return k_spmmv_pattern<VT, K, 4, false, 3, Acc>;
        else return k_spmmv_pattern<VT, K, 4, true, 2, Acc>;
    };
    return launch_short<VT>(pick(), h, X, ldx, Y, ldy, acc, vec, s);
}

// Unroll choices keep U * K <= 16 gathered values per thread.
template <class VT, int K, bool PIPE, class Acc>
cudaError_t pick_u(const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int acc, int vec,
                   cudaStream_t s) {
    const int u = h->unroll ? h->unroll : 4;
    if constexpr (K >= 8) {
        return u >= 2 ? run<VT, K, 2, PIPE, Acc>(h, X, ldx, Y, ldy, acc, vec, s)
                      : run<VT, K, 1, PIPE, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
    } else if constexpr (K >= 4) {
        if (u >= 4) return run<VT, K, 4, PIPE, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
        if (u >= 2) return run<VT, K, 2, PIPE, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
        return run<VT, K, 1, PIPE, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
    } else {
        if constexpr (K == 1 && PIPE) {
            constexpr int own = sizeof(VT) == 8 ? 2 : 4;  // the library's choice and its kernel (run_block)
            if (h->C == 32 && u == own)
                return launch_short<VT>(k_spmv_short<VT, own, true, Acc, 32>, h, X, ldx, Y, ldy, acc, vec, s);
        }
        if (u >= 8) return run<VT, K, 8, PIPE, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
        if (u >= 4) return run<VT, K, 4, PIPE, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
        if (u >= 2) return run<VT, K, 2, PIPE, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
        return run<VT, K, 1, PIPE, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
    }
}

// K columns: the long rows, then the short ones.  Launch mode 1 runs the
// software-pipelined chain at every block width.  Without sell_set_launch the
// chain is pipelined, with the unroll that was fastest or within 4 % of it on
// the matrices it was swept on (block 128; unroll 4 without pipelining, block
// 256 in brackets): binary64 at one vector unroll 2: 1M banded rows 66.9 us
// [92.2], 2M sorted lognormal rows 133 us [137]; binary32 at one vector unroll
// 4: 1M banded rows 33.2 us [36.8]; four vectors 4 (binary64 2): 1M lognormal
// rows binary32 98 us [131], 1M banded rows binary64 149 us [187]; eight
// vectors 2 (binary64 1): 1M lognormal rows binary32 105 us [117], binary64
// 219 us [269], 1M banded rows binary32 77 us [103].
template <class VT, int K, class Acc, class AccL>
cudaError_t run_block(const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int acc, int vec,
                      void *part, int32_t *cnt, int32_t *cnt2, cudaStream_t s) {
    if (h->nunits) {
        const cudaError_t e = run_long<VT, K, AccL>(h, X, ldx, Y, ldy, acc, vec, part, cnt, cnt2, s);
        if (e != cudaSuccess) return e;
    }
    if constexpr (K == 1) {
        if (ldx >= kWidePitch)
            return launch_short_with<VT, WidePitch>(k_spmv_short<VT, 1, false, Acc, 0, WidePitch>, h, X, ldx, Y, ldy, acc,
                                                    vec, s);
    }
    if constexpr (pattern_width<VT, K>()) {
        if (h->scol) return run_pattern<VT, K, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
    }
    // (launch mode 2 is the bulk-staged kernel's: its unroll counts slots)
    if ((h->pipeline != 0 && h->unroll == 0) || h->pipeline == 2) {
        if constexpr (K == 1) {
            if (h->C == 32)
                return launch_short<VT>(k_spmv_short<VT, sizeof(VT) == 8 ? 2 : 4, true, Acc, 32>, h, X, ldx, Y, ldy, acc,
                                        vec, s);
        }
        constexpr int U = K == 8 ? 2 : 4;
        if constexpr (K > 1 && sizeof(VT) == 8) {
            // Few rows like the loads in flight better than the warps, and so
            // do even ones at two vectors.  Unroll 4 (2 at eight vectors)
            // against half of it: two vectors, 280,000 lognormal rows sorted /
            // in windows of 256 / unsorted 36 / 68 / 111 and 43 / 80 / 123 us,
            // 1M sorted 72 and 70 us, 100^3 stencil 94 and 96 us; eight,
            // 280,000 lognormal rows 76 / 220 / 387 and 84 / 235 / 406 us, 1M
            // banded rows 408 and 401 us.  Four: 20,000 banded rows 12.3 and
            // 15.8 us, but 500^2 Laplacian 18 and 14 us, 200,000 sorted
            // lognormal rows 45 and 42 us.
            const bool even = !h->nunits;
            if (K == 4 ? even && h->nrows <= kFewRows / 8 : h->nrows <= kFewRows || (K == 2 && even))
                return run<VT, K, U, true, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
        }
        return run<VT, K, sizeof(VT) == 8 ? U / 2 : U, true, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
    }
    if (h->pipeline != 0) return pick_u<VT, K, true, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
    return pick_u<VT, K, false, Acc>(h, X, ldx, Y, ldy, acc, vec, s);
}

}  // namespace spmv_impl

// Launch one column block (kb in {1, 2, 4, 8}) of the given storage type and
// accumulation (AccL: of the rows over kSeg entries); part/cnt/cnt2 = nullptr
// uses the handle's scratch.  A single column with launch mode 2 goes to the
// bulk-staged kernel.
template <class VT, class Acc, class AccL = Acc>
cudaError_t spmv_block(const sell_matrix *h, const void *X, int64_t ldx, void *Y, int64_t ldy, int kb,
                       int acc, int vec, void *part, int32_t *cnt, int32_t *cnt2, cudaStream_t s) {
    using namespace spmv_impl;
    if constexpr (std::is_same<Acc, AccL>::value) {  // the bulk kernel has one accumulation for all rows
        if (!part && kb == 1 && h->pipeline == 2 && h->bulk_grid > 0)
            return bulk::run<VT, Acc>(h, X, ldx, Y, ldy, acc, s);
    }
    if (!part) {
        part = h->part;
        cnt = h->cnt;
        cnt2 = h->cnt2;
    }
    switch (kb) {
        case 1: return run_block<VT, 1, Acc, AccL>(h, X, ldx, Y, ldy, acc, vec, part, cnt, cnt2, s);
        case 2: return run_block<VT, 2, Acc, AccL>(h, X, ldx, Y, ldy, acc, vec, part, cnt, cnt2, s);
        case 4: return run_block<VT, 4, Acc, AccL>(h, X, ldx, Y, ldy, acc, vec, part, cnt, cnt2, s);
        default: return run_block<VT, 8, Acc, AccL>(h, X, ldx, Y, ldy, acc, vec, part, cnt, cnt2, s);
    }
}

}  // namespace sell
