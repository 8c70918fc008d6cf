"""The padded blocks' memory: refused, or asked for while the stream is captured,
the product takes the blocks 4, 2, 1 and gives the same bits; there before the
capture, the padded block is captured and replays right whatever widths run in
between.  (Matrices and widths that do run padded: binary32 at three and five
vectors, binary64 at seven.)"""
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu

LONG = synth.lognormal(3001, seed=1, cap=700)
SHORT = synth.banded(40000, seed=2)


class _Watched:
    """A torch-backed allocator that lists the requests while watching, and refuses those of `refuse` bytes."""

    def __init__(self):
        import torch
        from paper_1307_6209_gb300 import sell
        self.asked, self.watch, self.refuse, self.refused = [], False, None, 0

        def _alloc(nbytes, ctx, stream):
            if self.watch:
                self.asked.append(int(nbytes))
            if self.refuse is not None and nbytes == self.refuse:
                self.refused += 1
                return None
            return torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)

        def _free(ptr, ctx, stream):
            if ptr:
                torch.cuda.caching_allocator_delete(ptr)

        self.fns = sell.ALLOC_FN(_alloc), sell.FREE_FN(_free)

    def __enter__(self):
        from paper_1307_6209_gb300 import sell
        assert sell.load().sell_set_allocator(*self.fns, None) == sell.SELL_OK
        return self

    def __exit__(self, *e):
        from paper_1307_6209_gb300 import sell
        assert sell.load().sell_set_allocator(sell.ALLOC_FN(), sell.FREE_FN(), None) == sell.SELL_OK


def _columns(A, store, k, seed):
    """X and the product of each column alone."""
    import torch
    from paper_1307_6209_gb300 import sell
    dt = torch.float64 if store == 0 else torch.float32
    X = torch.from_numpy(synth.block(A.ncols, 8, seed=seed)).to(dt).cuda()
    h = sell.sell_build(A, C=7, store_type=store)
    cols = []
    for q in range(8):
        y = torch.empty(A.nrows, dtype=dt, device="cuda")
        sell.sell_spmv(h, X[:, q].contiguous(), y)
        cols.append(y)
    torch.cuda.synchronize()
    h.free()
    return X, torch.stack(cols, 1)


CASES = [(LONG, 1, 3), (LONG, 1, 5), (LONG, 0, 7), (SHORT, 1, 3), (SHORT, 1, 5), (SHORT, 0, 7)]
IDS = [f"{'long' if A is LONG else 'short'}-{'f64' if s == 0 else 'f32'}-{k}" for A, s, k in CASES]


@pytest.mark.parametrize("A,store,k", CASES, ids=IDS)
def test_refused_copy(A, store, k):
    import torch
    from paper_1307_6209_gb300 import sell
    X, want = _columns(A, store, k, 3)
    x = X[:, :k].contiguous()
    copy = A.ncols * 8 * X.element_size()
    with _Watched() as w:
        h = sell.sell_build(A, C=32, store_type=store)
        w.refuse, w.watch = copy, True
        for _ in range(2):
            y = torch.zeros((A.nrows, k), dtype=X.dtype, device="cuda")
            sell.sell_spmmv(h, x, y)
            torch.cuda.synchronize()
            assert torch.equal(y, want[:, :k])
        assert w.refused == 2
        w.refuse = None
        y = torch.zeros((A.nrows, k), dtype=X.dtype, device="cuda")
        sell.sell_spmmv(h, x, y)  # memory is back: padded from here on
        assert torch.equal(y, want[:, :k]) and w.asked.count(copy) == 3
        h.free()


@pytest.mark.parametrize("A,store,k", CASES, ids=IDS)
@pytest.mark.parametrize("warm", [False, True])
def test_captured(A, store, k, warm):
    import torch
    from paper_1307_6209_gb300 import sell
    X, want = _columns(A, store, k, 4)
    x, y = X[:, :k].contiguous(), torch.zeros((A.nrows, k), dtype=X.dtype, device="cuda")
    copy = A.ncols * 8 * X.element_size()
    with _Watched() as w:
        h = sell.sell_build(A, C=32, store_type=store)
        w.watch = True
        out = torch.empty((A.nrows, 8), dtype=X.dtype, device="cuda")
        sell.sell_spmmv(h, X, out)  # the long rows' scratch of unpadded blocks is at its widest
        if warm:
            sell.sell_spmmv(h, x, y)
        assert w.asked.count(copy) == int(warm)
        before = len(w.asked)
        torch.cuda.synchronize()
        s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            sell.sell_spmmv(h, x, y)
        assert len(w.asked) == before  # nothing is allocated under capture
        for m in (3, 7, 5, 8):
            z = torch.empty((A.nrows, m), dtype=X.dtype, device="cuda")
            sell.sell_spmmv(h, X[:, :m].contiguous(), z)
            assert torch.equal(z, want[:, :m])
        for _ in range(3):
            y.zero_()
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(y, want[:, :k])
        del g
        h.free()
