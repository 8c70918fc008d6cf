"""Blocks of 3 and 5 to 7 right-hand sides, which run as one block of 4 or 8
on a padded copy of X: every column has the bits of its product alone, with
short, long and pattern rows, dense and strided X and Y, accumulation, narrow
blocks asked for; nothing beside the columns is written or read; the first
such product inside a capture allocates nothing and replays right after other
widths have run."""
import numpy as np
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu

MATS = [("lognormal", synth.lognormal(3001, seed=1, cap=700)), ("banded", synth.banded(2000, seed=2)),
        ("stencil", synth.stencil27(20, 0.1, seed=3)), ("dense", synth.dense(130, 90)),
        ("wide", synth.random_csr(20, 300, density=0.03, seed=4))]  # too few entries for a pass over X


@pytest.mark.parametrize("store,flags", [(0, 0), (1, 0), (1, 2), (2, 8)])
@pytest.mark.parametrize("name,A", MATS, ids=[n for n, _ in MATS])
def test_odd_widths_keep_each_columns_bits(name, A, store, flags):
    import torch
    from paper_1307_6209_gb300 import sell
    dt = torch.float64 if store == 0 else torch.float32
    X, Y0 = (torch.from_numpy(synth.block(n, 23, seed=5)).to(dt).cuda() for n in (A.ncols, A.nrows))
    for C, sigma in [(32, 1), (7, 1), (64, 10 ** 9)]:
        h = sell.sell_build(A, C=C, sigma=sigma, store_type=store)
        want = {}
        for acc in (0, sell.SELL_SPMV_ACCUMULATE):
            cols = []
            for q in range(23):
                y = Y0[:, q].clone()
                sell.sell_spmv(h, X[:, q].contiguous(), y, flags=flags | acc)
                cols.append(y)
            want[acc] = torch.stack(cols, 1)
        for k in (3, 5, 6, 7, 11, 13, 23):
            for pad in (0, 2):
                for extra in (0, sell.SELL_SPMV_ACCUMULATE, sell.SELL_SPMV_RHS_BLOCK4, sell.SELL_SPMV_RHS_BLOCK2):
                    xs = torch.full((A.ncols, k + pad), float("nan"), dtype=dt, device="cuda")
                    ys = torch.full((A.nrows, k + pad), 7.0, dtype=dt, device="cuda")
                    xs[:, :k], ys[:, :k] = X[:, :k], Y0[:, :k]
                    sell.sell_spmmv(h, xs, ys, flags=flags | extra, k=k)
                    assert torch.equal(ys[:, :k], want[extra & 1][:, :k]), (C, k, pad, extra)
                    assert bool((ys[:, k:] == 7.0).all())
        h.free()


def test_captured_odd_width():
    import torch
    from paper_1307_6209_gb300 import sell
    A = MATS[0][1]
    X = torch.from_numpy(synth.block(A.ncols, 8, seed=6)).cuda()
    ref = sell.sell_build(A, C=7)
    want = torch.empty((A.nrows, 8), dtype=torch.float64, device="cuda")
    sell.sell_spmmv(ref, X, want)
    for warm in ((), (3,), (5, 3)):
        h = sell.sell_build(A, C=32)
        for k in warm + (8,):  # the long rows' scratch is at its widest before the capture
            sell.sell_spmmv(h, X[:, :k].contiguous(), torch.empty((A.nrows, k), dtype=torch.float64, device="cuda"))
        x5, y5 = X[:, :5].contiguous(), torch.zeros((A.nrows, 5), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            sell.sell_spmmv(h, x5, y5)
        for k in (7, 3, 8):
            sell.sell_spmmv(h, X[:, :k].contiguous(), torch.empty((A.nrows, k), dtype=torch.float64, device="cuda"))
        torch.cuda.synchronize()
        for _ in range(3):
            y5.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(y5, want[:, :5])
        h.free()


def test_failing_allocation_takes_the_narrow_blocks():
    import torch
    from paper_1307_6209_gb300 import sell
    A = MATS[1][1]  # no long rows: their scratch is needed either way
    X = torch.from_numpy(synth.block(A.ncols, 5, seed=7)).cuda()
    lib, state = sell.load(), {"fail": False}

    def _alloc(nbytes, ctx, stream):
        if state["fail"] and nbytes >= A.ncols * 64:
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)

    def _free(ptr, ctx, stream):
        if ptr:
            torch.cuda.caching_allocator_delete(ptr)

    a, f = sell.ALLOC_FN(_alloc), sell.FREE_FN(_free)
    assert lib.sell_set_allocator(a, f, None) == sell.SELL_OK
    try:
        got = []
        for fail in (False, True):
            h = sell.sell_build(A, C=32)
            state["fail"] = fail
            y = torch.zeros((A.nrows, 5), dtype=torch.float64, device="cuda")
            sell.sell_spmmv(h, X, y)
            got.append(y)
            state["fail"] = False
            h.free()
        assert torch.equal(*got)
    finally:
        assert lib.sell_set_allocator(sell.ALLOC_FN(), sell.FREE_FN(), None) == sell.SELL_OK


@pytest.mark.parametrize("store", [0, 1])
def test_padded_widths_leave_a_captured_graphs_scratch(store):
    """A graph of two columns, captured with the long rows' scratch at two:
    padded widths after it neither move nor free that scratch."""
    import torch
    from paper_1307_6209_gb300 import sell
    A = MATS[0][1]
    dt = torch.float64 if store == 0 else torch.float32
    X = torch.from_numpy(synth.block(A.ncols, 7, seed=8)).to(dt).cuda()
    h = sell.sell_build(A, C=32, store_type=store)
    x2, y2 = X[:, :2].contiguous(), torch.zeros((A.nrows, 2), dtype=dt, device="cuda")
    sell.sell_spmmv(h, x2, y2)
    want = y2.clone()
    torch.cuda.synchronize()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        sell.sell_spmmv(h, x2, y2)
    y7 = torch.zeros((A.nrows, 7), dtype=dt, device="cuda")
    sell.sell_spmmv(h, X, y7)
    if store:
        sell.sell_spmmv(h, X[:, :3].contiguous(), torch.zeros((A.nrows, 3), dtype=dt, device="cuda"))
    torch.cuda.synchronize()
    for _ in range(3):
        y2.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y2, want) and torch.equal(y7[:, :2], want)
    h.free()


def test_threads_on_one_stream_keep_their_padded_copies():
    import threading
    import torch
    from paper_1307_6209_gb300 import sell
    A = MATS[1][1]
    h = sell.sell_build(A, C=32, store_type=1)
    Xs = [torch.from_numpy(synth.block(A.ncols, 5, seed=20 + t)).float().cuda() for t in range(4)]
    ref = sell.sell_build(A, C=32, store_type=1)
    want = []
    for X in Xs:
        y = torch.empty((A.nrows, 5), device="cuda")
        sell.sell_spmmv(ref, X, y)
        want.append(y)
    ys = [[torch.zeros((A.nrows, 5), device="cuda") for _ in range(200)] for _ in Xs]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def work(t):
        with torch.cuda.stream(stream):
            for y in ys[t]:
                sell.sell_spmmv(h, Xs[t], y)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    torch.cuda.synchronize()
    assert all(torch.equal(y, w) for l, w in zip(ys, want) for y in l)
