"""The packed copies of chunks with few long rows: less than a quarter of the
chunks they come from, whatever the number of segments, and products with the
bits of chunk heights that have no such copies."""
import numpy as np
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


def _matrix(rl, ncols, seed):
    rng = np.random.default_rng(seed)
    rpt = np.concatenate([[0], np.cumsum(rl)])
    return synth.CSR(len(rl), ncols, rpt, rng.integers(0, ncols, rpt[-1]).astype(np.int32),
                     rng.standard_normal(int(rpt[-1])))


@pytest.mark.parametrize("store,value", [(0, 8), (1, 4), (2, 2)])
@pytest.mark.parametrize("length", [65, 128, 1000])
def test_a_slightly_long_row_in_every_chunk(length, store, value):
    from paper_1307_6209_gb300 import sell
    rl = np.full(32 * 200, 3)
    rl[::32] = length
    for C in (32, 128):
        h = sell.sell_build(_matrix(rl, 5000, 1), C=C, store_type=store)
        i, entry = h.info, value + 4
        nseg = -(-length // 64)
        units = i.nchunks * nseg
        # the format, the work lists and the sums' scratch, with a quarter of the format for the copies
        lists = i.nchunks * (4 + 4 * C + 12) + units * 8 + units * 32 + i.nchunks * C * 4 + units * C * (4 + 8)
        fixed = 8 * (i.nchunks + 1) + 8 * i.nchunks + 4 * i.nchunks * C
        assert i.device_bytes <= 1.25 * entry * i.stored + lists + fixed, (C, i.device_bytes, entry * i.stored)
        h.free()


@pytest.mark.parametrize("store,flags", [(0, 0), (1, 0), (1, 2), (2, 0)])
def test_every_number_of_packed_segments(store, flags):
    import torch
    from paper_1307_6209_gb300 import sell
    rl, chunk = [], np.full(32, 2)
    for m in range(1, 5):
        for nseg in list(range(2, 12)) + [16, 31, 32, 33]:
            c = chunk.copy()
            c[7 * np.arange(m) + 3] = nseg * 64 - np.arange(m) * 13 % 64
            rl.append(c)
    A = _matrix(np.concatenate(rl), 3000, 2)
    dt = torch.float64 if store == 0 else torch.float32
    X = torch.from_numpy(synth.block(A.ncols, 8, seed=3)).to(dt).cuda()
    want = {}
    for C in (7, 32, 64, 96):
        h = sell.sell_build(A, C=C, store_type=store)
        for k in (1, 2, 4, 8):
            Y = torch.full((A.nrows, k), float("nan"), dtype=dt, device="cuda")
            sell.sell_spmmv(h, X[:, :k].contiguous(), Y, flags=flags)
            got = Y.cpu().numpy().tobytes()
            assert got == want.setdefault(k, got), (C, k)
        h.free()
