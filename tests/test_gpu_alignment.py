"""An allocator whose pointers are aligned to 8 bytes and no more: matrices with
rows over 64 entries (work lists, packed entries, partial sums) build and
multiply to the same bits through every entry point, launch mode 2 refuses."""
import numpy as np
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


def _matrix():
    """Chunks with few long rows, with many, and rows over 16384 entries."""
    rng = np.random.default_rng(3)
    rl = np.full(400, 5)
    rl[[0, 33, 70, 399]] = 65, 17000, 200, 130
    rl[128:256] = rng.integers(60, 200, 128)
    rpt = np.concatenate([[0], np.cumsum(rl)])
    col = np.concatenate([np.sort(rng.choice(17000, n, replace=False)) for n in rl]).astype(np.int32)
    return synth.CSR(400, 17000, rpt, col, rng.standard_normal(int(rpt[-1])))


def _all_products(A, store, C, sigma):
    import torch
    from paper_1307_6209_gb300 import sell
    dt = torch.float64 if store == 0 else torch.float32
    X = torch.from_numpy(synth.block(A.ncols, 8, seed=4)).to(dt).cuda()
    out = []
    h = sell.sell_build(A, C=C, sigma=sigma, store_type=store)
    for k in (1, 2, 3, 4, 7, 8):
        x = X[:, :k].contiguous()
        for call in (sell.sell_spmmv, sell.sell_spmmv_noalloc):
            y = torch.full((A.nrows, k), float("nan"), dtype=dt, device="cuda")
            call(h, x, y)
            out.append(y)
        y = torch.full((A.nrows, k), float("nan"), dtype=dt, device="cuda")
        plan = sell.sell_batch_create([(h, x, y, 0)])
        plan.run()
        out.append(y)
        torch.cuda.synchronize()
        plan.free()
    return h, [y.cpu().numpy().tobytes() for y in out]


@pytest.mark.parametrize("store", [0, 1, 2])
@pytest.mark.parametrize("C,sigma", [(7, 1), (32, 1), (64, 10 ** 9), (96, 1)])
def test_eight_byte_pointers(C, sigma, store):
    import torch
    from paper_1307_6209_gb300 import sell
    A = _matrix()
    h, want = _all_products(A, store, C, sigma)
    h.free()
    lib, shifted = sell.load(), set()

    def _alloc(nbytes, ctx, stream):
        p = torch.cuda.caching_allocator_alloc(int(nbytes) + 16, torch.cuda.current_device(), stream or 0) + 8
        shifted.add(p)
        return p

    def _free(ptr, ctx, stream):
        if ptr:
            shifted.remove(ptr)
            torch.cuda.caching_allocator_delete(ptr - 8)

    a, f = sell.ALLOC_FN(_alloc), sell.FREE_FN(_free)
    assert lib.sell_set_allocator(a, f, None) == sell.SELL_OK
    try:
        h, got = _all_products(A, store, C, sigma)
        with pytest.raises(sell.SellError) as e:
            sell.sell_set_launch(h, 0, 0, 2)
        assert e.value.status == sell.SELL_EUNSUPPORTED
        assert shifted
        h.free()
        assert got == want
    finally:
        assert lib.sell_set_allocator(sell.ALLOC_FN(), sell.FREE_FN(), None) == sell.SELL_OK
