"""sell_spmv_dot's forms (a thread, a warp, a block per range) give the
documented order of additions bit for bit, at the lengths where the form
changes and in between, in binary64 and binary32, behind every kind of
product, again and again."""
import numpy as np
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


def _fma_exact(a, b, c):
    from fractions import Fraction
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def _documented(x, y):
    n = len(x)
    ln = -(-n // 1024)
    part = np.zeros(1024)
    for b in range(1024):
        red = np.zeros(256)
        for t in range(256):
            s = 0.0
            for i in range(b * ln + t, min(n, (b + 1) * ln), 256):
                s = _fma_exact(float(x[i]), float(y[i]), s)
            red[t] = s
        w = 128
        while w:
            red[:w] = red[:w] + red[w:2 * w]
            w //= 2
        part[b] = red[0]
    w = 512
    while w:
        part[:w] = part[:w] + part[w:2 * w]
        w //= 2
    return part[0]


def _diag(n, long_row):
    rl = np.ones(n, np.int64)
    if long_row:
        rl[n // 2] = min(n, 100)
    rpt = np.concatenate([[0], np.cumsum(rl)])
    col = np.concatenate([np.arange(n // 2), np.arange(rl[n // 2]) if long_row else [n // 2],
                          np.arange(n // 2 + 1, n)]).astype(np.int32)
    return synth.CSR(n, n, rpt, col, np.random.default_rng(n).standard_normal(int(rpt[-1])))


@pytest.mark.parametrize("store", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 1000, 1024, 1025, 4096, 8191, 8192, 8193, 40000, 262143, 262144, 262145, 300001])
def test_dot_order(n, store):
    import torch
    from paper_1307_6209_gb300 import sell
    dt = torch.float64 if store == 0 else torch.float32
    xd = torch.from_numpy(synth.vector(n, seed=n)).to(dt).cuda()
    want = None
    for A in (_diag(n, False), _diag(n, True)):
        h = sell.sell_build(A, C=32, store_type=store)
        y, dot = torch.empty(n, dtype=dt, device="cuda"), torch.empty(3, dtype=torch.float64, device="cuda")
        for i in range(3):
            sell.sell_spmv_dot(h, xd, y, dot[i:])
        got = dot.cpu().numpy()
        want = _documented(xd.cpu().double().numpy(), y.cpu().double().numpy())
        assert np.all(got == want), (n, got, want)
        h.free()
