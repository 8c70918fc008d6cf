"""Edges of the tiled scatter and of the sorts in sell_build, byte for byte
against the oracle's build: rows around the tile (16 columns) and segment (64)
widths, slices wider than their chunk neighbours, a chunk height that is a
multiple of 32 but no power of two, column permutation, window lengths that
are and are not powers of two, keys of one to four digit passes."""
import numpy as np
import pytest

import oracle
from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


def _rows(lengths, ncols, seed):
    rng = np.random.default_rng(seed)
    rl = np.asarray(lengths, np.int64)
    rpt = np.concatenate([[0], np.cumsum(rl)])
    col = np.concatenate([np.sort(rng.choice(ncols, n, replace=False)) for n in rl] or [np.zeros(0)]).astype(np.int32)
    return synth.CSR(len(rl), ncols, rpt, col, rng.standard_normal(int(rpt[-1])))


def _compare(A, C, sigma, store=0, permute=False):
    from paper_1307_6209_gb300 import sell
    h = sell.sell_build(A, C=C, sigma=sigma, store_type=store, flags=sell.SELL_BUILD_PERMUTE_COLS if permute else 0)
    G, F = sell.sell_export(h), oracle.sell_build(A, C, sigma, permute_cols=permute)
    for k in ("cs", "cl", "srl", "perm", "col"):
        assert G[k].tobytes() == F[k].tobytes(), (k, C, sigma)
    ref = F["val"] if store == 0 else oracle.round_values(F["val"], store)
    assert G["val"].tobytes() == ref.tobytes()
    h.free()


@pytest.mark.parametrize("C", [32, 64, 96, 160])
@pytest.mark.parametrize("store", [0, 1, 2])
def test_rows_around_the_tile_edges(C, store):
    lens = [0, 1, 15, 16, 17, 31, 33, 63, 64, 65, 127, 128, 129, 700]
    rng = np.random.default_rng(C)
    A = _rows(rng.choice(lens, 400), 701, seed=C + store)
    for sigma in (1, 96, 10 ** 9):
        _compare(A, C, sigma, store)


@pytest.mark.parametrize("C", [32, 96])
def test_column_permutation_with_long_rows(C):
    lens = np.random.default_rng(5).integers(0, 200, 333)
    _compare(_rows(lens, 333, seed=7), C, 10 ** 9, permute=True)


@pytest.mark.parametrize("sigma", [2, 3, 32, 64, 100, 1000, 2048, 4095, 4096])
@pytest.mark.parametrize("N", [2, 63, 4097, 10001])
def test_window_lengths(N, sigma):
    rng = np.random.default_rng(N + sigma)
    _compare(_rows(rng.integers(0, 6, N), 50, seed=sigma), 32, sigma)


@pytest.mark.parametrize("N,cap,sigma", [(4200, 3, 10 ** 9), (9000, 300, 5000), (70000, 40, 4100),
                                         (300000, 5, 4097), (6000, 5000, 10 ** 9)])
def test_radix_digit_passes(N, cap, sigma):
    rng = np.random.default_rng(N)
    rl = rng.integers(0, min(cap, 6) + 1, N)
    rl[rng.integers(0, N, 3)] = cap  # the longest row sets the key's width
    _compare(_rows(rl, max(cap, 10), seed=cap), 32, sigma)


def test_bad_columns_are_refused_in_every_path():
    """Column indices are checked while the entries are scattered: short rows,
    a long row's later segment, chunk heights of both scatter kernels, with
    the column permutation (which looks the index up)."""
    from paper_1307_6209_gb300 import sell
    A = _rows(np.where(np.arange(300) == 150, 250, 3), 300, seed=3)
    for at in (0, int(A.rpt[150]) + 249, A.nnz - 1):
        for bad in (-1, 300, 2 ** 31 - 1):
            B = synth.CSR(A.nrows, A.ncols, A.rpt, A.col.copy(), A.val)
            B.col[at] = bad
            for C in (7, 32, 64):
                for flags in (0, sell.SELL_BUILD_PERMUTE_COLS):
                    with pytest.raises(sell.SellError) as e:
                        sell.sell_build(B, C=C, sigma=64, flags=flags)
                    assert e.value.status == sell.SELL_EINVAL and "column index" in str(e.value)
