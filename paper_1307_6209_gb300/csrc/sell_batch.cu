// sell_batch.cu -- many SELL-C-sigma products in few launches.
//
// A plan splits every product into column blocks of 8, 4, 2 or 1 right-hand
// sides (at most the item's SELL_SPMV_RHS_BLOCK* width) and groups the blocks
// by kernel variant (value type, block width, plain or compensated
// accumulation).  Each variant present gets one launch for its products' long
// rows and one for their short rows (per 144 products): the products and the
// block ranges of their work travel in the kernel's parameter space -- a unit
// is one block's worth of sorted rows of one product (128 by default, 64 or
// 256 after sell_batch_set_launch), or as many threads of its long-row work
// (sell_long.cuh).  Creating a plan makes one device allocation (the
// products' long-row scratch) and no copies, and does not synchronise.  One
// block per unit, biggest products first; the hardware block scheduler
// balances the uneven products.  The launches of a plan do not depend on each
// other: each is a programmatic dependent of the one before, so that its
// blocks start as soon as all blocks of that one have started, and a last
// block waits for the end of the launch before, so that the plan has ended
// when its last launch has.  (A grid-stride "persistent" form of this kernel
// was measured: its loop-carried state raised the register count from 40 to
// 64, cut the resident blocks per SM from 6 to 4 and made the batch slower.)
//
// Every row is computed by the same per-row arithmetic as sell_spmmv
// (sell_rowdot.cuh), so a product's result is bit-identical whether it runs
// alone or inside any batch.
#include <algorithm>
#include <map>
#include <new>
#include <tuple>
#include <type_traits>
#include <vector>

#include "sell_long.cuh"
#include "sell_rowdot.cuh"

namespace sell {
namespace {

constexpr int kTileRows = 256;

// One product's short rows, and its long rows.
struct RowProd {
    const void *val;
    const int32_t *col;
    const int64_t *cs;
    const int32_t *srl, *perm;
    const void *X;
    void *Y;
    int64_t ldx, ldy, N;
    int32_t C, acc, vec;
    Pitch pitch;  // ldx in bytes (unless it is wide)
};
struct LongProd {
    LongArgs a;
    const void *val, *lval;
    void *part;    // this product's own segment scratch (owned by the plan)
    int32_t *cnt;  // ... segment counters
    int32_t *cnt2; // ... group counters
    const void *X;
    void *Y;
    int64_t ldx, ldy;
    int32_t acc, vec;
    Pitch pitch;
};

template <class LD, class P>
__device__ __forceinline__ LD pitch_of(const P &p) {
    if constexpr (std::is_same<LD, Pitch>::value) return p.pitch;
    else return p.ldx;
}

// The products of one launch travel in the kernel's parameter space (read
// through the constant cache when a unit needs a field), which keeps the
// register footprint at that of the single-product kernel.  The work units
// need no table: block w belongs to product i with start[i] <= w <
// start[i+1], tile threads per block.
constexpr int kLaunchProds = 144;  // 144 * 216 B + the ranges fit the 32 KB parameter limit

template <class P>
struct LaunchParams {
    P prods[kLaunchProds];
    int32_t start[kLaunchProds + 1];
    int32_t nprod;
};
using RowParams = LaunchParams<RowProd>;
using LongParams = LaunchParams<LongProd>;
static_assert(sizeof(RowParams) <= 32764 && sizeof(LongParams) <= 32764, "kernel parameter limit");

// The product of block w, or -1 past the last unit (those threads wait for
// the launch before this one).
template <class P>
__device__ __forceinline__ int product_of(const LaunchParams<P> &lp, int32_t w) {
    if (w >= lp.start[lp.nprod]) {
        wait_for_predecessor();
        return -1;
    }
    int lo = 0, hi = lp.nprod;  // last range with start <= w
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (lp.start[mid] <= w) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Unroll and resident blocks (of 256 threads) of the short rows' kernels,
// software pipelined at every width.  CT is 32 where every chunk of the
// launch's products is 32 rows high -- the strides are then constants of the
// load instructions, which at one vector of 4-byte values saves the spills of
// the 32-register form (every warp slot of the SM) -- else 0.  Measured
// against the kernels that held both the long and the short rows, binary32
// unless stated: 48 banded matrices one vector 138 -> 131 us (CT 0 with 40
// registers 144, with 32 and spills 158-182), 96 mixed matrices 386 -> 361 us;
// two vectors, compensated, 145 -> 144 us; four 349 -> 335 us; eight 402 ->
// 402 us (48 mixed), 347 -> 337 us (48 banded); binary64 one vector 242 ->
// 196 us, two 187 -> 177 us, four 309 -> 307 us, eight 453 -> 441 us;
// bfloat16 114 -> 99 us.  Narrower caps spill (binary32 at eight vectors with
// 6 blocks 489 us, binary64 at one vector with 8 blocks 235 us).
struct RowShape {
    int unroll, blocks;
};
template <class VT, int K, int CT>
constexpr RowShape row_shape() {
    if (sizeof(VT) == 8) return K == 1 ? RowShape{4, 6} : K == 2 ? RowShape{2, 4} : K == 4 ? RowShape{2, 4} : RowShape{2, 3};
    return K == 1 ? (CT ? RowShape{4, 8} : RowShape{4, 6}) : K == 2 ? RowShape{4, 5} : K == 4 ? RowShape{4, 5} : RowShape{2, 4};
}

template <class VT, int K, class Acc, int CT, class LD = Pitch>
__global__ void __launch_bounds__(kTileRows, (row_shape<VT, K, CT>().blocks))
k_batch_rows(const __grid_constant__ RowParams lp) {
    using XT = typename XType<VT>::T;
    dependents_may_start();
    const int i = product_of(lp, (int32_t)blockIdx.x);
    if (i < 0) return;
    const RowProd &P = lp.prods[i];
    const int64_t r = (int64_t)((int32_t)blockIdx.x - lp.start[i]) * blockDim.x + threadIdx.x;
    if (r < P.N)
        short_row<VT, XT, K, row_shape<VT, K, CT>().unroll, true, Acc, false, CT>(
            static_cast<const VT *>(P.val), P.col, P.cs, P.srl, P.perm, Pattern{}, static_cast<const XT *>(P.X),
            pitch_of<LD>(P), static_cast<XT *>(P.Y), P.ldy, P.C, (uint32_t)r, P.acc, P.vec, l2_evict_first_policy());
}

template <class VT, int K, class AccL, class LD = Pitch>
__global__ void __launch_bounds__(kTileRows) k_batch_long(const __grid_constant__ LongParams lp) {
    using XT = typename XType<VT>::T;
    constexpr LongShape S = long_shape<VT, K>();
    dependents_may_start();
    const int i = product_of(lp, (int32_t)blockIdx.x);
    if (i < 0) return;
    const LongProd &P = lp.prods[i];
    long_rows<VT, K, S.unroll, S.pipe, AccL, false>(static_cast<const VT *>(P.val), static_cast<const VT *>(P.lval), P.a,
                                              P.part, P.cnt, P.cnt2, static_cast<const XT *>(P.X), pitch_of<LD>(P),
                                              static_cast<XT *>(P.Y), P.ldy, P.acc, P.vec,
                                              (int64_t)((int32_t)blockIdx.x - lp.start[i]) * blockDim.x + threadIdx.x);
}

using RowFn = void (*)(const RowParams);
using LongFn = void (*)(const LongParams);

// kb 0: one column of an X with a wide pitch.  c32: every chunk height is 32.
template <class VT, class Acc>
RowFn row_fn(int kb, bool c32) {
    switch (kb) {
        case 0: return k_batch_rows<VT, 1, Acc, 0, WidePitch>;
        case 1: return c32 ? k_batch_rows<VT, 1, Acc, 32> : k_batch_rows<VT, 1, Acc, 0>;
        case 2: return c32 ? k_batch_rows<VT, 2, Acc, 32> : k_batch_rows<VT, 2, Acc, 0>;
        case 4: return c32 ? k_batch_rows<VT, 4, Acc, 32> : k_batch_rows<VT, 4, Acc, 0>;
        default: return c32 ? k_batch_rows<VT, 8, Acc, 32> : k_batch_rows<VT, 8, Acc, 0>;
    }
}
template <class VT, class Acc>
LongFn long_fn(int kb) {
    switch (kb) {
        case 0: return k_batch_long<VT, 1, Acc, WidePitch>;
        case 1: return k_batch_long<VT, 1, Acc>;
        case 2: return k_batch_long<VT, 2, Acc>;
        case 4: return k_batch_long<VT, 4, Acc>;
        default: return k_batch_long<VT, 8, Acc>;
    }
}

// comp: 0 binary32 chains, 1 Dot2 on every row, 2 Dot2 on the long rows only.
RowFn row_kernel(int type, int comp, int kb, bool c32) {
    if (type == SELL_F64) return row_fn<double, Plain<double>>(kb, c32);
    if (type == SELL_F32) return comp == 1 ? row_fn<float, Dot2>(kb, c32) : row_fn<float, Plain<float>>(kb, c32);
    return comp == 1 ? row_fn<__nv_bfloat16, Dot2>(kb, c32) : row_fn<__nv_bfloat16, Plain<float>>(kb, c32);
}
LongFn long_kernel(int type, int comp, int kb) {
    if (type == SELL_F64) return long_fn<double, Plain<double>>(kb);
    if (type == SELL_F32) return comp ? long_fn<float, Dot2>(kb) : long_fn<float, Plain<float>>(kb);
    return comp ? long_fn<__nv_bfloat16, Dot2>(kb) : long_fn<__nv_bfloat16, Plain<float>>(kb);
}

}  // namespace

namespace {
size_t up256(size_t x) { return (x + 255) / 256 * 256; }
}  // namespace

// Long-row scratch of one batch item (all its column blocks): the segment
// partials of every block, then the counters of every block (cleared
// together).  0 for matrices without long rows.
size_t batch_item_scratch(const sell_matrix *h, int32_t k, uint32_t flags, size_t *counter_offset) {
    size_t pb = 0, cb = 0;
    if (h->nunits > 0 && h->nrows > 0) {
        for (int32_t done = 0; done < k;) {
            const int kb = rhs_block(k - done, max_rhs_block(flags));
            pb += up256((size_t)h->nunits * h->C * kb * 8);
            cb += up256((size_t)(h->nlong + h->nunits) * h->C * sizeof(int32_t));
            done += kb;
        }
    }
    if (counter_offset) *counter_offset = pb;
    return pb + cb;
}

namespace {
// An item's flags, with columns taken one at a time where X's pitch is wide.
uint32_t block_flags(const sell_batch_item &it) {
    return it.ldx < kWidePitch ? it.flags : it.flags | SELL_SPMV_RHS_BLOCK1;
}

// A product as the plan is put together.
struct Prod {
    RowProd row;
    LongProd lng;
    int32_t type, comp, kb;
    int64_t long_threads;
};

// The block ranges of a launch's products for blocks of `tile` threads.
// Returns the number of blocks.
int64_t threads_of(const RowProd &p) { return p.N; }
int64_t threads_of(const LongProd &p) { return p.a.lwork ? p.a.nwork * 32 : p.a.nwork * p.a.C; }
template <class P>
int64_t assign_units(LaunchParams<P> *lp, int tile) {
    int64_t w = 0;
    for (int j = 0; j < lp->nprod; ++j) {
        lp->start[j] = (int32_t)std::min<int64_t>(w, 0x7FFFFFFE);
        w += (threads_of(lp->prods[j]) + tile - 1) / tile;
    }
    lp->start[lp->nprod] = (int32_t)std::min<int64_t>(w, 0x7FFFFFFE);
    return w;
}
int64_t assign_units(void *params, bool lng, int tile) {
    return lng ? assign_units(static_cast<LongParams *>(params), tile) : assign_units(static_cast<RowParams *>(params), tile);
}
void delete_params(void *params, bool lng) {
    if (lng) delete static_cast<LongParams *>(params);
    else delete static_cast<RowParams *>(params);
}
constexpr int64_t kMaxUnits = 0x7FFFFFFE;  // and the block that waits

// Adds the launches of the products ids (at most kLaunchProds each) to the
// plan; what(id) gives a product's part of them.
template <class P, class What>
sell_status add_launches(sell_batch *b, void *fn, bool lng, const std::vector<int32_t> &ids, What what) {
    for (size_t p0 = 0; p0 < ids.size(); p0 += kLaunchProds) {
        const int np = (int)(std::min(ids.size(), p0 + (size_t)kLaunchProds) - p0);
        auto *lp = new (std::nothrow) LaunchParams<P>();
        if (!lp) return fail(SELL_ENOMEM, "sell_batch_create: host allocation failed");
        lp->nprod = np;
        for (int j = 0; j < np; ++j) lp->prods[j] = what(ids[p0 + j]);
        const int64_t w = assign_units(lp, b->tile);
        if (w == 0 || w > kMaxUnits) {
            delete lp;
            if (w == 0) continue;
            return fail(SELL_EUNSUPPORTED, "sell_batch_create: too many work units in one launch");
        }
        sell_batch::Group G;
        G.fn = fn;
        G.params = lp;
        G.lng = lng;
        G.nwork = w;
        G.grid = (int32_t)w;  // one block per unit
        b->groups.push_back(G);
        b->nwork += w;
    }
    return SELL_OK;
}
}  // namespace

sell_status batch_create(const sell_batch_item *items, int32_t n, cudaStream_t s, sell_batch *b,
                         void *const *scratch) {
    std::vector<Prod> prods;
    std::vector<const sell_matrix *> owner;
    b->al = current_allocator();
    // each item with long rows gets its own scratch (given by the caller, or
    // one allocation for the whole plan), so products of one plan -- even on
    // the same matrix -- never share segment partials or counters
    char *own = nullptr;
    if (!scratch) {
        size_t total = 0;
        for (int32_t i = 0; i < n; ++i)
            if (items[i].A && items[i].k >= 1)
                total += batch_item_scratch(items[i].A, items[i].k, block_flags(items[i]), nullptr);
        if (total > 0) {
            own = static_cast<char *>(b->al.get(total, s));
            if (!own) return fail(SELL_ENOMEM, "sell_batch_create: segment scratch allocation failed");
            b->scratch.push_back(own);
        }
    }
    size_t own_off = 0;
    for (int32_t i = 0; i < n; ++i) {
        const sell_batch_item &it = items[i];
        const sell_matrix *h = it.A;
        if (!h) return fail(SELL_EINVAL, "sell_batch_create: NULL matrix");
        if (it.k < 1 || it.ldx < it.k || it.ldy < it.k)
            return fail(SELL_EINVAL, "sell_batch_create: need k >= 1, ldx >= k, ldy >= k");
        if (h->nrows > 0 && (!it.X || !it.Y)) return fail(SELL_EINVAL, "sell_batch_create: NULL X/Y");
        if (it.flags & ~(SELL_SPMV_ACCUMULATE | kCompFlags | kRhsFlags))
            return fail(SELL_EINVAL, "sell_batch_create: unsupported flags");
        if ((it.flags & kCompFlags) && h->store_type == SELL_F64)
            return fail(SELL_EUNSUPPORTED, "compensated accumulation needs F32/BF16 storage");
        if (h->nrows == 0) continue;
        size_t coff = 0;
        const size_t sbytes = batch_item_scratch(h, it.k, block_flags(it), &coff);
        char *sc = nullptr;
        if (sbytes > 0) {
            sc = scratch ? static_cast<char *>(scratch[i]) : own + own_off;
            own_off += scratch ? 0 : sbytes;
            if (!sc) return fail(SELL_EINVAL, "sell_batch_create: missing scratch");
            SELL_CUDA_TRY(cudaMemsetAsync(sc + coff, 0, sbytes - coff, s));
        }
        size_t poff = 0, cpos = coff;
        const size_t xs = h->store_type == SELL_F64 ? 8 : 4;
        for (int32_t done = 0; done < it.k;) {
            const int kb = rhs_block(it.k - done, max_rhs_block(block_flags(it)));
            Prod P = {};
            RowProd &R = P.row;
            LongProd &L = P.lng;
            R.val = L.val = h->val;
            R.col = h->col;
            R.cs = h->cs;
            R.srl = h->srl;
            R.perm = (h->flags & SELL_BUILD_PERMUTE_COLS) ? nullptr : h->perm;
            R.N = h->nrows;
            R.C = h->C;
            L.a = long_args(h, false);
            L.lval = h->lval;
            if (sc) {
                L.part = sc + poff;
                L.cnt = reinterpret_cast<int32_t *>(sc + cpos);
                L.cnt2 = L.cnt + h->nlong * h->C;
                poff += up256((size_t)h->nunits * h->C * kb * 8);
                cpos += up256((size_t)(h->nlong + h->nunits) * h->C * sizeof(int32_t));
            }
            P.long_threads = long_threads(h);
            R.X = L.X = static_cast<const char *>(it.X) + done * xs;
            R.Y = L.Y = static_cast<char *>(it.Y) + done * xs;
            R.ldx = L.ldx = it.ldx;
            R.pitch = L.pitch = Pitch{(int32_t)(it.ldx * (int64_t)xs)};
            R.ldy = L.ldy = it.ldy;
            R.acc = L.acc = (it.flags & SELL_SPMV_ACCUMULATE) ? 1 : 0;
            R.vec = L.vec = x_vec(R.X, it.ldx, xs) | (x_vec(R.Y, it.ldy, xs) << 2);
            P.kb = it.ldx < kWidePitch ? kb : 0;
            P.type = h->store_type;
            P.comp = h->store_type != SELL_F64 ? comp_mode(it.flags) : 0;
            prods.push_back(P);
            owner.push_back(h);
            done += kb;
        }
    }
    // group by kernel variant; inside a group biggest first.  The long rows'
    // accumulation differs from the short rows' with COMPENSATED_LONG, so the
    // two kinds of launches are grouped apart
    int dev = 0;
    SELL_CUDA_TRY(cudaGetDevice(&dev));
    b->device = dev;
    b->nprod = (int32_t)prods.size();
    b->nwork = 0;
    std::vector<int32_t> ids(prods.size());
    for (size_t i = 0; i < ids.size(); ++i) ids[i] = (int32_t)i;
    std::stable_sort(ids.begin(), ids.end(),
                     [&](int32_t a, int32_t c) { return owner[a]->stored > owner[c]->stored; });
    struct Key {
        int type, comp, kb, c32;
        bool operator<(const Key &o) const {
            return std::tie(type, comp, kb, c32) < std::tie(o.type, o.comp, o.kb, o.c32);
        }
    };
    auto launches = [&](bool lng) -> sell_status {
        std::map<Key, std::vector<int32_t>> groups;
        for (int32_t id : ids) {
            const Prod &P = prods[id];
            if (lng && P.long_threads == 0) continue;
            const int c32 = !lng && P.kb > 0 && P.row.C == 32;
            groups[Key{P.type, lng ? (P.comp ? 1 : 0) : (P.comp == 1 ? 1 : 0), P.kb, c32}].push_back(id);
        }
        std::vector<std::pair<int64_t, Key>> order;  // biggest group first
        for (auto &kv : groups) {
            int64_t work = 0;
            for (int32_t id : kv.second) work += lng ? prods[id].long_threads : prods[id].row.N * std::max(1, prods[id].kb);
            order.push_back({work, kv.first});
        }
        std::stable_sort(order.begin(), order.end(), [](const std::pair<int64_t, Key> &a, const std::pair<int64_t, Key> &c) {
            return a.first > c.first;
        });
        for (auto &o : order) {
            const Key &k = o.second;
            if (lng) {
                void *fn = reinterpret_cast<void *>(long_kernel(k.type, k.comp, k.kb));
                SELL_TRY(add_launches<LongProd>(b, fn, true, groups[k], [&](int32_t id) { return prods[id].lng; }));
            } else {
                void *fn = reinterpret_cast<void *>(row_kernel(k.type, k.comp, k.kb, k.c32));
                SELL_TRY(add_launches<RowProd>(b, fn, false, groups[k], [&](int32_t id) { return prods[id].row; }));
            }
        }
        return SELL_OK;
    };
    SELL_TRY(launches(true));
    return launches(false);
}

void batch_release(sell_batch *b, cudaStream_t s) {
    for (auto &G : b->groups) delete_params(G.params, G.lng);
    b->groups.clear();
    for (void *p : b->scratch) b->al.put(p, s);
    b->scratch.clear();
}

sell_status batch_set_tile(sell_batch *b, int32_t tile) {
    if (tile != 64 && tile != 128 && tile != 256)
        return fail(SELL_EINVAL, "sell_batch_set_launch: block must be 64, 128 or 256");
    for (const sell_batch::Group &G : b->groups) {
        const int64_t w = assign_units(G.params, G.lng, tile);
        if (w > kMaxUnits) {
            for (const sell_batch::Group &H : b->groups) assign_units(H.params, H.lng, b->tile);
            return fail(SELL_EUNSUPPORTED, "sell_batch_set_launch: too many work units in one launch");
        }
    }
    b->tile = tile;
    b->nwork = 0;
    for (sell_batch::Group &G : b->groups) {
        G.nwork = assign_units(G.params, G.lng, tile);
        G.grid = (int32_t)G.nwork;
        b->nwork += G.nwork;
    }
    return SELL_OK;
}

sell_status batch_run(sell_batch *b, int32_t grid, cudaStream_t s) {
    if (grid != 0) return fail(SELL_EINVAL, "sell_batch_run: grid must be 0 (one block per work unit)");
    b->last_stream = s;
    b->ran = true;
    bool first = true;
    for (const sell_batch::Group &G : b->groups) {
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)G.grid + (first ? 0 : 1));  // the block that waits for the launch before
        cfg.blockDim = dim3(b->tile);
        cfg.stream = s;
        cfg.attrs = at;
        cfg.numAttrs = first ? 0 : 1;
        void *args[] = {G.params};
        SELL_CUDA_TRY(cudaLaunchKernelExC(&cfg, G.fn, args));
        first = false;
    }
    return SELL_OK;
}

}  // namespace sell
