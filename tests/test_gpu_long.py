"""Rows longer than 64 entries of single products, which run in a kernel of
their own ahead of the short rows': bit for bit the same for chunk heights that
are a multiple of 32 (virtual warps, packed entries for chunks with few long
rows) and that are not (units), at the edges of segments (64), groups (16384)
and the switch between the two forms (8 m <= C); ordered before whatever
follows on the stream, and capturable."""
import numpy as np
import pytest

import oracle
from paper_1307_6209_gb300 import synth
from tests.gpu_util import tol_f64

pytestmark = pytest.mark.gpu


def _matrix(lengths, ncols, seed):
    rng = np.random.default_rng(seed)
    rl = np.asarray(lengths, np.int64)
    rpt = np.concatenate([[0], np.cumsum(rl)])
    col = np.concatenate([np.sort(rng.choice(ncols, n, replace=False)) for n in rl]).astype(np.int32)
    return synth.CSR(len(rl), ncols, rpt, col, rng.standard_normal(int(rpt[-1])))


def _cases():
    rng = np.random.default_rng(0)
    few = np.full(200, 3)
    few[[0, 31, 40, 130, 199]] = [65, 64, 16384, 16385, 40000]
    edge = np.full(384, 5)  # exactly 4 of 32, 5 of 32, 12 of 96, 13 of 96 long rows per chunk
    edge[0:4], edge[32:37], edge[96:108], edge[192:205] = 100, 129, 70, 1000
    many = rng.integers(1, 400, 300)
    return [("few", _matrix(few, 40001, 1)), ("edge", _matrix(edge, 1200, 2)), ("many", _matrix(many, 500, 3)),
            ("all", _matrix(np.full(70, 700), 701, 4))]


CASES = _cases()


@pytest.mark.parametrize("store,flags", [(0, 0), (1, 0), (1, 2), (1, 8), (2, 8)])
@pytest.mark.parametrize("name,A", CASES, ids=[n for n, _ in CASES])
def test_long_rows_keep_the_bits(name, A, store, flags):
    import torch
    from paper_1307_6209_gb300 import sell
    X, Y0 = synth.block(A.ncols, 11, seed=5), synth.block(A.nrows, 11, seed=6)
    dt = torch.float64 if store == 0 else torch.float32
    Xd = torch.from_numpy(X).to(dt).cuda()
    want = {}
    for C, sigma in [(7, 1), (32, 1), (32, 10 ** 9), (64, 1), (96, 1), (96, 64), (128, 10 ** 9)]:
        h = sell.sell_build(A, C=C, sigma=sigma, store_type=store)
        for k in (1, 2, 4, 11):
            for acc in (0, sell.SELL_SPMV_ACCUMULATE):
                for rep in range(2):  # the counters are back at zero after a product
                    Y = torch.from_numpy(Y0[:, :k]).to(dt).cuda().contiguous()
                    sell.sell_spmmv(h, Xd[:, :k].contiguous(), Y, flags=flags | acc)
                    got = Y.cpu().numpy().tobytes()
                    assert got == want.setdefault((k, acc), got), (C, sigma, k, acc, rep)
        h.free()


@pytest.mark.parametrize("name,A", CASES, ids=[n for n, _ in CASES])
def test_long_rows_are_ordered_on_the_stream_and_captured(name, A):
    """A kernel that follows the product reads finished long rows, a kernel
    ahead of it has written x, products follow each other; the same in a
    captured graph."""
    import torch
    from paper_1307_6209_gb300 import sell
    x = synth.vector(A.ncols, seed=7)
    h = sell.sell_build(A, C=32, sigma=1)
    s = torch.cuda.Stream()
    xd, xs = torch.zeros(A.ncols, dtype=torch.float64, device="cuda"), torch.from_numpy(x).cuda()
    y, z = torch.empty(A.nrows, dtype=torch.float64, device="cuda"), torch.empty(A.nrows, dtype=torch.float64, device="cuda")
    ref, tol = oracle.csr_spmv(A, x), tol_f64(A.row_lengths(), oracle.csr_absdot(A, x))

    def step():
        xd.zero_()
        xd.add_(xs)
        sell.sell_spmv(h, xd, y)
        z.copy_(y)
        y.fill_(float("nan"))
        sell.sell_spmv(h, xd, y)
        z.add_(y)

    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        for _ in range(20):
            step()
        s.synchronize()
        assert np.all(np.abs(z.cpu().numpy() / 2 - ref) <= tol)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            step()
        for _ in range(5):
            z.fill_(0)
            g.replay()
        s.synchronize()
    assert np.all(np.abs(z.cpu().numpy() / 2 - ref) <= tol)
