"""Rows of X further apart than 2^31 bytes: such products run one column at a
time in kernels with 64-bit row pitches, single and batched, with short and
long rows, and give the bits of the same product on a dense X; the pitch just
below takes the usual kernels.  (X has two rows, so that it fits.)"""
import numpy as np
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ldx", [(1 << 28) - 8, 1 << 28, (1 << 28) + 3])
@pytest.mark.parametrize("k", [1, 3])
def test_wide_row_pitch(ldx, k):
    import torch
    from paper_1307_6209_gb300 import sell
    rng = np.random.default_rng(k)
    rl = rng.integers(0, 3, 200)
    rl[[3, 150]] = 300  # long rows (columns repeat: CRS allows it)
    rpt = np.concatenate([[0], np.cumsum(rl)])
    A = synth.CSR(200, 2, rpt, rng.integers(0, 2, rpt[-1]).astype(np.int32), rng.standard_normal(rpt[-1]))
    X = torch.from_numpy(synth.block(2, k, seed=1)).float().cuda()
    big = torch.zeros(ldx + 64, dtype=torch.float32, device="cuda")
    Xw = big.as_strided((2, k), (ldx, 1))
    Xw.copy_(X)
    for C in (7, 32, 64):
        h = sell.sell_build(A, C=C, store_type=sell.SELL_F32)
        want, got = (torch.zeros((200, k), device="cuda") for _ in range(2))
        sell.sell_spmmv(h, X, want)
        sell.sell_spmmv(h, Xw, got)
        assert torch.equal(got, want)
        got.zero_()
        sell.sell_spmmv_noalloc(h, Xw, got)
        assert torch.equal(got, want)
        got.zero_()
        plan = sell.sell_batch_create([(h, Xw, got, 0)])
        plan.run()
        assert torch.equal(got, want)
        plan.free()
        h.free()


def test_batch_of_all_forms_is_each_product_alone():
    """One plan over every value type, width and chunk height, more products
    than one launch takes, with and without long rows; block sizes changed;
    in a graph; right after and right before other work on the stream."""
    import torch
    from paper_1307_6209_gb300 import sell
    items, alone = [], []
    for i in range(300):
        A = synth.lognormal(60 + 7 * i, seed=i, cap=40 if i % 3 else 400)
        store = (sell.SELL_F32, sell.SELL_F64, sell.SELL_BF16)[0 if i < 160 else i % 3]
        k = 1 if i < 160 else (1, 2, 3, 4, 8, 9)[i % 6]
        h = sell.sell_build(A, C=(32, 64, 7, 96)[i % 4], sigma=(1, 10 ** 9)[i % 2], store_type=store)
        dt = torch.float64 if store == sell.SELL_F64 else torch.float32
        X = torch.from_numpy(synth.block(A.ncols, k, seed=i)).to(dt).cuda()
        fl = 0 if store == sell.SELL_F64 else (0, sell.SELL_SPMV_COMPENSATED, sell.SELL_SPMV_COMPENSATED_LONG)[i % 3]
        want = torch.empty((A.nrows, k), dtype=dt, device="cuda")
        sell.sell_spmmv(h, X, want, flags=fl)
        alone.append(want)
        items.append((h, X, torch.empty_like(want), fl))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    plan = sell.sell_batch_create(items, stream=s)

    def check(run):
        with torch.cuda.stream(s):
            for _, _, Y, _ in items:
                Y.fill_(float("nan"))
            run()
            out = [Y.clone() for _, _, Y, _ in items]
        s.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(out, alone))

    for block in (64, 128, 256):
        plan.set_launch(block)
        check(lambda: plan.run(stream=s))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        plan.run(stream=s)
        plan.run(stream=s)
    check(g.replay)
