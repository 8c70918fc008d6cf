"""sell_spmv_dot whose first call on a handle is captured in a graph: the call
allocates nothing, so calls outside the graph before its first replay, the
replays and calls after them all give the bits of a handle that was never
captured."""
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", [0, 1])
@pytest.mark.parametrize("name,A", [("warps", synth.laplace2d(64)), ("blocks", synth.laplace2d(520)),
                                    ("long", synth.long_row(9001, 9001, short_len=4, at=10, seed=2))],
                         ids=["warps", "blocks", "long"])
def test_first_dot_under_capture(name, A, store):
    import torch
    from paper_1307_6209_gb300 import sell
    dt = torch.float64 if store == 0 else torch.float32
    x = torch.from_numpy(synth.vector(A.ncols, seed=1)).to(dt).cuda()
    y = torch.empty(A.nrows, dtype=dt, device="cuda")
    want, got = (torch.empty(1, dtype=torch.float64, device="cuda") for _ in range(2))
    ref = sell.sell_build(A, C=32, store_type=store)
    sell.sell_spmv_dot(ref, x, y, want)
    torch.cuda.synchronize()

    # every allocation after the build is refused
    lib, state = sell.load(), {"refuse": False, "asked": 0}

    def _alloc(nbytes, ctx, stream):
        state["asked"] += state["refuse"]
        if state["refuse"]:
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)

    def _free(ptr, ctx, stream):
        if ptr:
            torch.cuda.caching_allocator_delete(ptr)

    a, f = sell.ALLOC_FN(_alloc), sell.FREE_FN(_free)
    for own in (False, True):
        if own:
            assert lib.sell_set_allocator(a, f, None) == sell.SELL_OK
        try:
            h = sell.sell_build(A, C=32, store_type=store)
            state["refuse"] = own
            torch.cuda.synchronize()
            s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                sell.sell_spmv_dot(h, x, y, got)
            for step in ("eager", "replay", "replay", "eager"):
                got.fill_(float("nan"))
                if step == "replay":
                    g.replay()
                else:
                    sell.sell_spmv_dot(h, x, y, got)
                torch.cuda.synchronize()
                assert torch.equal(got, want), (own, step)
            assert state["asked"] == 0
            del g
            state["refuse"] = False
            h.free()
        finally:
            if own:
                assert lib.sell_set_allocator(sell.ALLOC_FN(), sell.FREE_FN(), None) == sell.SELL_OK
