"""Products of matrices whose 32-row slices have one column pattern (the
columns then come from per-slice offsets): bit for bit the same as the general
kernels' -- which a chunk height that is no multiple of 32 selects -- and
within the oracle's bound.  Grids around the slice width, dense blocks around
the segment width, slices with and without a pattern in one matrix, several
slices per chunk, sorted rows, column permutation, every number of right-hand
sides, strided X and Y, accumulation."""
import numpy as np
import pytest

import oracle
from paper_1307_6209_gb300 import synth
from tests.gpu_util import tol_f64

pytestmark = pytest.mark.gpu


def _mixed(n):
    """Dense rows, diagonal rows, empty rows and random rows, 96 of each."""
    rng = np.random.default_rng(n)
    rows = []
    for r in range(384):
        kind = r // 96
        rows.append(np.arange(n) if kind == 0 else np.array([r % n, (r % n) + 3]) % n if kind == 1
                    else np.zeros(0, int) if kind == 2 else rng.choice(n, 5, replace=False))
    rl = np.array([len(c) for c in rows])
    return synth.CSR(384, n, np.concatenate([[0], np.cumsum(rl)]), np.concatenate(rows).astype(np.int32),
                     rng.standard_normal(int(rl.sum())))


MATS = [("stencil33", synth.stencil27(33, 0.1, seed=1)), ("stencil64", synth.stencil27(64, 0.1, seed=2)),
        ("laplace100x40", synth.laplace2d(100, 40)), ("dense63", synth.dense(63)), ("dense64", synth.dense(64, 64)),
        ("dense130", synth.dense(130, 65)), ("dense300x700", synth.dense(300, 700)), ("mixed", _mixed(200))]


def _product(h, X, k, flags=0, Y0=None, pad=0):
    import torch
    from paper_1307_6209_gb300 import sell
    dt = h.value_dtype
    n, m = h.info.ncols, h.info.nrows
    Xd = torch.zeros((n, k + pad), dtype=dt, device="cuda")
    Xd[:, :k] = torch.from_numpy(X[:, :k]).to(dt)
    Yd = torch.zeros((m, k + pad), dtype=dt, device="cuda")
    if Y0 is not None:
        Yd[:, :k] = torch.from_numpy(Y0[:, :k]).to(dt)
    sell.sell_spmmv(h, Xd, Yd, flags=flags, k=k)
    return Yd[:, :k].cpu().numpy()


@pytest.mark.parametrize("store,comp", [(0, 0), (1, 0), (1, 2), (1, 8), (2, 0), (2, 2)])
@pytest.mark.parametrize("name,A", MATS, ids=[n for n, _ in MATS])
def test_pattern_products_keep_the_bits(name, A, store, comp):
    from paper_1307_6209_gb300 import sell
    X, Y0 = synth.block(A.ncols, 11, seed=3), synth.block(A.nrows, 11, seed=4)
    ref = sell.sell_build(A, C=7, sigma=1, store_type=store)
    for C, sigma in [(32, 1), (64, 1), (96, 10 ** 9), (128, 64)]:
        h = sell.sell_build(A, C=C, sigma=sigma, store_type=store)
        for k in (1, 2, 3, 4, 8, 11):
            for pad in (0, 1, 4):
                for flags, y0 in [(comp, None), (comp | sell.SELL_SPMV_ACCUMULATE, Y0)]:
                    got, want = (_product(m, X, k, flags, y0, pad) for m in (h, ref))
                    assert got.tobytes() == want.tobytes(), (C, sigma, k, pad, flags)
        h.free()
    ref.free()


@pytest.mark.parametrize("name,A", MATS[:6], ids=[n for n, _ in MATS[:6]])
def test_pattern_product_is_the_oracles(name, A):
    import torch
    from paper_1307_6209_gb300 import sell
    x = synth.vector(A.ncols, seed=5)
    for C in (32, 64):
        h = sell.sell_build(A, C=C)
        y = torch.empty(A.nrows, dtype=torch.float64, device="cuda")
        for block in (32, 128, 512):
            sell.sell_set_launch(h, block)
            y.fill_(float("nan"))
            sell.sell_spmv(h, torch.from_numpy(x).cuda(), y)
            err = np.abs(y.cpu().numpy() - oracle.csr_spmv(A, x))
            assert np.all(err <= tol_f64(A.row_lengths(), oracle.csr_absdot(A, x)))


def test_pattern_with_permuted_columns_and_special_values():
    """P A P^T of a grid, and infinities and NaN in x outside a row's columns
    (no entry of that row may touch them)."""
    import torch
    from paper_1307_6209_gb300 import sell
    A = synth.stencil27(40, 0.1, seed=6)
    a = sell.sell_build(A, C=32, sigma=256, flags=sell.SELL_BUILD_PERMUTE_COLS)
    b = sell.sell_build(A, C=7, sigma=256, flags=sell.SELL_BUILD_PERMUTE_COLS)
    X = synth.block(A.ncols, 1, seed=7)
    assert _product(a, X, 1).tobytes() == _product(b, X, 1).tobytes()
    h = sell.sell_build(A, C=32)
    x = synth.vector(A.ncols, seed=8)
    x[0], x[20000] = np.inf, np.nan
    y = torch.empty(A.nrows, dtype=torch.float64, device="cuda")
    sell.sell_spmv(h, torch.from_numpy(x).cuda(), y)
    rows = np.repeat(np.arange(A.nrows), A.row_lengths())
    hit = np.unique(rows[np.isin(A.col, [0, 20000])])
    assert np.array_equal(np.nonzero(~np.isfinite(y.cpu().numpy()))[0], hit)


@pytest.mark.parametrize("sigma", [1, 256, 10 ** 9])
@pytest.mark.parametrize("which", ["val", "col", "all"])
def test_arrays_off_the_16_byte_grid_take_the_general_kernel(which, sigma):
    """An allocator may return a pointer that is aligned for its values only:
    the kernels that prefetch in 16-byte units are not used then."""
    import torch
    from paper_1307_6209_gb300 import sell
    A = synth.dense(1000, 60)
    x = torch.from_numpy(synth.block(A.ncols, 1, seed=4)[:, 0].copy()).cuda()
    h = sell.sell_build(A, C=32, sigma=sigma)
    want = torch.zeros(A.nrows, dtype=torch.float64, device="cuda")
    sell.sell_spmv(h, x, want)
    size = sell.sell_info(h).stored * (8 if which == "val" else 4)
    h.free()
    lib, shifted = sell.load(), []

    def _alloc(nbytes, ctx, stream):
        p = torch.cuda.caching_allocator_alloc(int(nbytes) + 16, torch.cuda.current_device(), stream or 0)
        if which == "all" or nbytes == size:
            p += 8
            shifted.append(p)
        return p

    def _free(ptr, ctx, stream):
        if ptr and ptr in shifted:
            shifted.remove(ptr)
            ptr -= 8
        if ptr:
            torch.cuda.caching_allocator_delete(ptr)

    a, f = sell.ALLOC_FN(_alloc), sell.FREE_FN(_free)
    assert lib.sell_set_allocator(a, f, None) == sell.SELL_OK
    try:
        h = sell.sell_build(A, C=32, sigma=sigma)
        assert which == "all" or len(shifted) == 1
        y = torch.zeros_like(want)
        sell.sell_spmv(h, x, y)
        assert torch.equal(y, want)
        h.free()
    finally:
        assert lib.sell_set_allocator(sell.ALLOC_FN(), sell.FREE_FN(), None) == sell.SELL_OK
