"""The tuner at several right-hand sides: the pipelined launches and the
library's own are among its candidates (so that what it returns was not slower
than an untuned handle where both were timed), and the tuned handle keeps the
bits.  At one right-hand side the library's own launch is one of the sweep."""
import pytest

from paper_1307_6209_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store,k", [(0, 8), (1, 8), (1, 4), (1, 3), (0, 1), (1, 1)])
def test_candidates_hold_the_untuned_launch(store, k):
    import torch
    from paper_1307_6209_gb300 import autotune, sell
    A = synth.lognormal_device(50000, seed=5)
    r = autotune.tune(A, store_type=store, k=k, Cs=(32,), sigmas=(4096,), keep=1, reps=5, cache=None)
    us = {(c["block"], c["unroll"], c["pipeline"]): c["us"] for c in r.launches}
    own = (0, 0, -1) if k > 1 else (128, 2 if store == 0 else 4, 1)
    assert {p for _, _, p in us} >= {0, 1} and own in us
    assert r.best.us == us[(r.best.block, r.best.unroll, r.best.pipeline)] == min(us.values())
    tuned = autotune.build_tuned(A, r.best, store_type=store)
    plain = sell.sell_build(A, C=32, sigma=4096, store_type=store)
    dt = torch.float64 if store == 0 else torch.float32
    X = torch.rand((A.ncols, k), dtype=dt, device="cuda")
    Y = [torch.empty((A.nrows, k), dtype=dt, device="cuda") for _ in range(2)]
    sell.sell_spmmv(tuned, X, Y[0])
    sell.sell_spmmv(plain, X, Y[1])
    assert torch.equal(*Y)
