"""device_bytes counts the padded copy of X and its scratch once they are there,
and a server takes them as resident."""
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store,k", [(0, 7), (1, 3), (1, 5)])
@pytest.mark.parametrize("name,A", [("short", synth.banded(40000, seed=2)), ("long", synth.lognormal(3001, seed=1, cap=700))],
                         ids=["short", "long"])
def test_padded_copy_is_counted(name, A, store, k):
    import torch
    from paper_1307_6209_gb300 import sell
    dt, word = (torch.float64, 8) if store == 0 else (torch.float32, 4)
    h = sell.sell_build(A, C=32, store_type=store)
    built = h.info.device_bytes
    X, Y = (torch.zeros((n, 8), dtype=dt, device="cuda") for n in (A.ncols, A.nrows))
    sell.sell_spmmv(h, X, Y)
    assert sell.sell_info(h).device_bytes == built  # eight columns are a block of their own
    for _ in range(2):
        sell.sell_spmmv(h, X[:, :k].contiguous(), Y[:, :k].contiguous())
        more = sell.sell_info(h).device_bytes - built
        rl = A.row_lengths()
        units = sum(-(-int(rl[c:c + 32].max()) // 64) for c in range(0, A.nrows, 32) if rl[c:c + 32].max() > 64)
        assert more == A.ncols * 8 * word + units * 32 * 64
    srv = sell.sell_server_create([h], built + more + (1 << 20), 4, 2)
    assert sell.sell_server_stats(srv)["resident_bytes"] == built + more
    sell.sell_server_destroy(srv)
    torch.cuda.synchronize()
    h.free()
