"""The fold of a long row's partial sums at several right-hand sides: the
columns' additions run side by side, not one after another (eight binary32
vectors cost less than two products of one), and every column keeps the bits
of its own product, for one completed row per warp, a few and many."""
import numpy as np
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


def _us(h, X, Y):
    import torch
    from paper_1307_6209_gb300 import sell
    best = 1e9
    for _ in range(8):
        sell.sell_spmmv(h, X, Y)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            sell.sell_spmmv(h, X, Y)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 50)
    return best


def test_columns_fold_side_by_side():
    import torch
    from paper_1307_6209_gb300 import sell
    A = synth.long_row(10000, 10000, short_len=3, at=77, seed=1)
    h = sell.sell_build(A, C=32, store_type=sell.SELL_F32)
    us = {}
    for k in (1, 8):
        X = torch.from_numpy(synth.block(A.ncols, k, seed=2)).float().cuda()
        us[k] = _us(h, X, torch.empty((A.nrows, k), dtype=torch.float32, device="cuda"))
    assert us[8] < 2 * us[1], us


@pytest.mark.parametrize("store,flags", [(0, 0), (1, 0), (1, 2), (2, 8)])
@pytest.mark.parametrize("rows", [1, 2, 3, 5, 8, 9, 32])
@pytest.mark.parametrize("length", [65, 64 * 17, 64 * 33 + 1])
def test_completed_rows_per_warp(rows, length, store, flags):
    import torch
    from paper_1307_6209_gb300 import sell
    rng = np.random.default_rng(rows)
    rl = np.full(96, 2)
    rl[32:32 + rows] = length + np.arange(rows) % 3 * 64
    rpt = np.concatenate([[0], np.cumsum(rl)])
    A = synth.CSR(96, 3000, rpt, rng.integers(0, 3000, rpt[-1]).astype(np.int32), rng.standard_normal(int(rpt[-1])))
    h = sell.sell_build(A, C=32, store_type=store)
    dt = torch.float64 if store == 0 else torch.float32
    X = torch.from_numpy(synth.block(A.ncols, 8, seed=3)).to(dt).cuda()
    cols = []
    for q in range(8):
        y = torch.empty(A.nrows, dtype=dt, device="cuda")
        sell.sell_spmv(h, X[:, q].contiguous(), y, flags=flags)
        cols.append(y)
    want = torch.stack(cols, 1)
    for k in (2, 4, 8):
        for _ in range(3):  # whichever warp completes a row
            Y = torch.empty((A.nrows, k), dtype=dt, device="cuda")
            sell.sell_spmmv(h, X[:, :k].contiguous(), Y, flags=flags)
            assert torch.equal(Y, want[:, :k])
