"""The rows of a ragged last warp run beside the long rows' kernel and not
after it: a product whose row count is no multiple of 32 takes the time of
the same product with empty rows up to the next multiple."""
import numpy as np
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


def _matrix(n):
    """A long row (segments that take a while to fold), and 16 rows of 64 entries at the end of 2000."""
    rl = np.zeros(n, np.int64)
    rl[5], rl[1984:2000] = 16000, 64
    rpt = np.concatenate([[0], np.cumsum(rl)])
    rng = np.random.default_rng(1)
    return synth.CSR(n, 2000, rpt, rng.integers(0, 2000, rpt[-1]).astype(np.int32), rng.standard_normal(int(rpt[-1])))


def test_ragged_last_warp_does_not_wait():
    import torch
    from paper_1307_6209_gb300 import sell
    X = torch.from_numpy(synth.block(2000, 8, seed=2)).cuda()
    hs = [(sell.sell_build(_matrix(n), C=32), torch.empty((n, 8), dtype=torch.float64, device="cuda"))
          for n in (2000, 2016)]
    best = [1e9, 1e9]
    for _ in range(10):
        for i, (h, Y) in enumerate(hs):
            sell.sell_spmmv(h, X, Y)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                sell.sell_spmmv(h, X, Y)
            b.record()
            b.synchronize()
            best[i] = min(best[i], a.elapsed_time(b))
    assert torch.equal(hs[0][1], hs[1][1][:2000])
    # waiting adds the rows' own time, about a third of the long row's
    assert best[0] <= 1.15 * best[1], best
