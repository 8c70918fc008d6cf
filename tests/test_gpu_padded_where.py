"""Which matrices run odd widths as a padded block: by the entries per column,
and more of them where neighbouring rows' columns lie close together (device_bytes
counts the padded copy).  Either way every column has the bits of its product
alone."""
import numpy as np
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu

N = 150000


def _matrix(kind, w):
    rng = np.random.default_rng(w)
    if kind == "random":
        col = rng.integers(0, N, (N, w))
    else:  # a band whose columns follow no pattern
        col = np.clip(np.arange(N)[:, None] + np.sort(rng.integers(-32, 32, (N, w)), axis=1), 0, N - 1)
    return synth.CSR(N, N, np.arange(N + 1, dtype=np.int64) * w, col.reshape(-1).astype(np.int32),
                     rng.standard_normal(N * w))


@pytest.mark.parametrize("kind,w,k,padded", [
    ("random", 2, 5, False), ("random", 2, 7, True), ("random", 4, 3, True), ("random", 4, 5, True),
    ("band", 4, 5, False), ("band", 12, 3, False), ("band", 12, 6, False), ("band", 4, 7, False), ("band", 6, 7, True),
    ("band", 18, 3, True), ("band", 18, 5, True)])
@pytest.mark.parametrize("store", [1, 2])
def test_padded_or_not(kind, w, k, padded, store):
    import torch
    from paper_1307_6209_gb300 import sell
    A = _matrix(kind, w)
    h = sell.sell_build(A, C=32, store_type=store)
    X = torch.from_numpy(synth.block(N, k, seed=1)).float().cuda()
    Y = torch.empty((N, k), device="cuda")
    sell.sell_spmmv(h, X, Y)
    assert (sell.sell_info(h).device_bytes > h.info.device_bytes) == padded
    for q in range(k):
        y = torch.empty(N, device="cuda")
        sell.sell_spmv(h, X[:, q].contiguous(), y)
        assert torch.equal(Y[:, q], y)
    h.free()
