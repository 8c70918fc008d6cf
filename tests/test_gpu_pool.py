"""The library's memory pool: sell_free keeps at most 1 GiB of it (and at
most 1/128 of the device's memory) for the next build, sell_set_allocator
returns all that is unused, and memory that is kept is used again."""
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


def test_pool_is_bounded_reused_and_given_back():
    import torch
    from paper_1307_6209_gb300 import sell

    def used():
        torch.cuda.synchronize()
        free, total = torch.cuda.mem_get_info()
        return total - free

    def give_back():
        sell.use_torch_allocator(False)

    small, big = synth.stencil27_device(30), synth.stencil27_device(170)  # big: 131 M entries, 1.6 GB as a handle
    sell.sell_build(small).free()  # the pool exists
    give_back()
    torch.cuda.empty_cache()
    base = used()
    bound = min(1 << 30, torch.cuda.mem_get_info()[1] // 128) + (64 << 20)
    h, g = sell.sell_build(big), sell.sell_build(small)
    assert used() - base > h.info.device_bytes
    h.free()
    kept = used() - base
    assert kept <= bound + g.info.device_bytes
    peak = 0
    for _ in range(3):  # builds that fit in what is kept map nothing
        h = sell.sell_build(small)
        peak = max(peak, used() - base)
        h.free()
    assert peak <= kept
    g.free()
    assert used() - base <= bound
    give_back()
    assert used() - base <= 8 << 20
