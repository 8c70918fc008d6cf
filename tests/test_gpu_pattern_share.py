"""Which matrices keep column offsets beside their columns: those with at least
half of their entries in slices that are read by one pattern.  A slice whose
first 64 columns have a pattern and whose others have none counts as a whole,
and rows of one or two entries do not count."""
import numpy as np
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


def _csr(cols, ncols):
    """Rows of equal length."""
    n, w = cols.shape
    return synth.CSR(n, ncols, np.arange(n + 1, dtype=np.int64) * w, cols.reshape(-1).astype(np.int32),
                     np.random.default_rng(w).standard_normal(n * w))


def _bytes(A):
    from paper_1307_6209_gb300 import sell
    h = sell.sell_build(A, C=32)
    b = h.info.device_bytes
    h.free()
    return b


def test_a_slice_counts_as_a_whole():
    rng = np.random.default_rng(0)
    n, w = 640, 192
    random = rng.integers(0, 5000, (n, w))
    head = random.copy()
    head[:, :128] = np.arange(n)[:, None] + np.arange(128)
    whole = np.arange(n)[:, None] + np.arange(w)
    plain = _bytes(_csr(random, 5000))
    assert _bytes(_csr(head, 5000)) == plain
    assert _bytes(_csr(whole, 5000)) > plain  # offsets


@pytest.mark.parametrize("width", [1, 2, 3])
def test_rows_with_next_to_no_columns(width):
    n = 3200
    plain = 12 * n * width + 8 * (n // 32 + 1) + 8 * (n // 32) + 4 * n
    got = _bytes(_csr(np.arange(n)[:, None] + np.arange(width), n + width))
    assert (got == plain) if width < 3 else (got > plain)


def test_products_keep_the_bits():
    import torch
    from paper_1307_6209_gb300 import sell
    rng = np.random.default_rng(1)
    n = 960
    rl = rng.integers(0, 3, n)
    rl[320:640] = 70  # pattern slices with long rows between slices of short rows
    start = np.concatenate([[0], np.cumsum(rl)])
    col = np.concatenate([r + np.arange(k) for r, k in enumerate(rl)]).astype(np.int32)
    A = synth.CSR(n, n + 80, start, col, rng.standard_normal(int(start[-1])))
    X = torch.from_numpy(synth.block(A.ncols, 8, seed=2)).cuda()
    got = []
    for C in (7, 32, 64):
        h = sell.sell_build(A, C=C)
        for k in (1, 2, 8):
            y = torch.empty((n, k), dtype=torch.float64, device="cuda")
            sell.sell_spmmv(h, X[:, :k].contiguous(), y)
            got.append(y.cpu().numpy().tobytes())
        h.free()
    assert got[:3] == got[3:6] == got[6:]
